// sort.cuh -- stable tile sort (sort.cu).
#pragma once
#include "pic_internal.cuh"
#include "push.cuh"

namespace pic {

size_t sort_scratch_bytes(long long cap);
size_t scan_scratch_words(long long m);
void scan_exclusive(const uint32_t *in, uint32_t *out, long long m, uint32_t *scratch, cudaStream_t st);
// a sort's outcome in its scratch: the permutation (new -> old), the sorted
// keys and the number of entries (device)
struct SortResult {
    const uint32_t *perm, *key;
    const long long *neff;
};
SortResult sort_by_tile(const uint32_t *cell, long long n, const long long *dcount, const Grid &g, void *scratch,
                        cudaStream_t st);
// the particle arrays in sorted order (dead ones dropped), starts[0..ntiles]
// and *dcount (the live particles)
template <class P_t>
void sort_apply(const P_t &src, const P_t &dst, const SortResult &r, long long n, const Grid &g, uint32_t *starts,
                long long *dcount, cudaStream_t st);

}  // namespace pic
