"""What a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``listed()`` names the standard ones,
``draw(rng)`` gives others of the same ranges, ``prepare(case, seed)`` builds
what a program has in hand before the call (a loaded simulation, or the inputs
of a run), ``run(state)`` is one pass through the public entry points of
``paper_2104_00642_gb300.pic``, ``work(case)`` counts the bytes and operations
a pass cannot do without, and ``exact(case, seed)`` is the same pass in plain
64-bit torch.

Kinds of case:

* ``plasma``: a uniform thermal plasma (or the cold Langmuir oscillation) in
  1D, 2D or 3D, all axes periodic: the bulk of any run.
* ``foil``: a slab hit by a laser that enters through the absorbing x-min face.
* ``qed``: fast electrons in a strong uniform magnetic field with photon
  emission and pair creation (tables or the surrogate networks).
* ``cascade``: a whole short run of single-electron cascades by Method II:
  create, load, step, read the particles, destroy.
* ``train``: training of a surrogate network.

Outputs: the field components come as borrowed views of the resident arrays in
the simulation's own precision; energies come from the diagnostics (the Gauss
residual, which is round-off around zero, is left out).  Particles are returned
where their order does not hang on a rounding: in the FP64 form, and in the
cascades, which never sort (momenta only: in a uniform field shared by all
replicas positions mean nothing).  In the FP32 form a particle within a
rounding of a cell face changes places with its neighbours at the next sort,
so there J, E, B and the energies stand for the particles.
"""
import math

import numpy as np
import torch

from paper_2104_00642_gb300 import pic, workloads as W

TWO_PI = 2.0 * math.pi
M_PROTON = 1836.15267343
MEC2_KEV = 510.99895
COMPS = ("Ex", "Ey", "Ez", "Bx", "By", "Bz", "Jx", "Jy", "Jz")
PREC = {"f32": pic.FP32_CELLOFF, "f64": pic.FP64_PLAIN}


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the 1D Langmuir oscillation, logged every 10 steps: a few thousand
        # particles, where launches and round trips are all there is
        dict(name="langmuir_1d", kind="plasma", dim=1, nx=256, ny=1, nz=1, dx=0.05, ppc=100, T_keV=0.0, amp=0.01,
             prec="f32", order=2, sort=0, steps=10, log=True, dump=False),
        # a hot 2D plasma stepped between snapshots: energies, all field
        # components and the charge density to the host
        dict(name="thermal_2d_snapshot", kind="plasma", dim=2, nx=256, ny=256, nz=1, dx=0.1, ppc=16, T_keV=100.0,
             amp=0.0, prec="f32", order=2, sort=8, steps=8, log=True, dump=True),
        # the laser-foil production run (Sec. III(a)) while the pulse comes up
        # to the slab: 4.2 million particles, half the grid in vacuum
        dict(name="laser_foil_2d", kind="foil", nx=2048, ny=1024, slab0=1024, slab1=1088, ppc=32, a0=20.0,
             prec="f32", sort=16, steps=32, particles=False),
        # the same physics in the plain FP64 form, phase space read at the end
        dict(name="laser_foil_2d_f64", kind="foil", nx=512, ny=256, slab0=256, slab1=288, ppc=32, a0=20.0,
             prec="f64", sort=16, steps=16, particles=True),
        # a hot 3D plasma: the largest particle count of the set
        dict(name="thermal_3d", kind="plasma", dim=3, nx=128, ny=128, nz=128, dx=0.1, ppc=8, T_keV=200.0, amp=0.0,
             prec="f32", order=2, sort=4, steps=4, log=False, dump=False),
        # 3D on a grid of odd sizes
        dict(name="thermal_3d_odd", kind="plasma", dim=3, nx=61, ny=45, nz=39, dx=0.1, ppc=8, T_keV=200.0, amp=0.0,
             prec="f32", order=2, sort=4, steps=8, log=False, dump=False),
        # the self-heating study (Sec. III(b)) with the order-4 shape, logged
        dict(name="self_heating_2d_order4", kind="plasma", dim=2, nx=128, ny=128, nz=1, dx=TWO_PI / 320, ppc=16,
             T_keV=1.0, amp=0.0, prec="f32", order=4, sort=16, steps=16, log=True, dump=False),
        # strong-field QED in 2D (the collision's beam energy and cell size,
        # chi ~ 1), photons above 10 MeV kept, rates from the tables
        dict(name="qed_2d_table", kind="qed", dim=2, nx=512, ny=256, nz=1, electrons=1 << 20, gamma0=1957.0, B0=200.0,
             mode="table", sort=8, steps=8),
        # the same with the surrogate networks
        dict(name="qed_2d_surrogate", kind="qed", dim=2, nx=512, ny=256, nz=1, electrons=1 << 20, gamma0=1957.0,
             B0=200.0, mode="surrogate", sort=8, steps=8),
        # the same in 3D (tables)
        dict(name="qed_3d_table", kind="qed", dim=3, nx=48, ny=48, nz=48, electrons=200_000, gamma0=1957.0, B0=200.0,
             mode="table", sort=8, steps=8),
        # replicas of the cascade of Fig. 9 (Method II), a whole short run
        dict(name="cascade_method2", kind="cascade", replicas=2000, gamma0=1000.0, b=0.009, steps=350),
        # a stretch of the training of the emission network
        dict(name="train_emission_net", kind="train", process=0, batch=16384, iterations=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plasma", "plasma", "plasma", "foil", "qed", "qed", "cascade", "train"])
    if kind == "plasma":
        dim = rng.choice([1, 2, 2, 3, 3])
        prec = rng.choice(["f32", "f32", "f32", "f64"])
        order = 4 if dim < 3 and rng.random() < 0.3 else 2
        n = [1, 1, 1]
        lo, hi = {1: (64, 4096), 2: (48, 768), 3: (20, 128)}[dim]
        for d in range(dim):
            n[d] = _log_int(rng, lo, hi)
            if rng.random() < 0.5:
                n[d] = max(16, n[d] // 16 * 16)  # round sizes half of the time
        cells = n[0] * n[1] * n[2]
        most = 2_000_000 if prec == "f64" else (8_000_000 if order == 2 else 2_000_000)
        ppc = max(1, min(_log_int(rng, 2, 100 if dim == 1 else 32), most // cells))
        return dict(kind=kind, dim=dim, nx=n[0], ny=n[1], nz=n[2], dx=round(rng.uniform(0.03, 0.15), 4), ppc=ppc,
                    T_keV=round(rng.uniform(150.0, 600.0), 1), amp=0.0, prec=prec, order=order,
                    sort=rng.choice([4, 8, 16]), steps=rng.choice([1, 4, 8, 16]), log=rng.random() < 0.4, dump=False)
    if kind == "foil":
        prec = rng.choice(["f32", "f32", "f64"])
        nx, ny = (_log_int(rng, 256, 2048), _log_int(rng, 100, 1024)) if prec == "f32" else \
                 (_log_int(rng, 200, 600), _log_int(rng, 64, 256))
        width = max(4, nx // rng.choice([8, 16, 32]))
        ppc = rng.choice([8, 16, 25, 32])
        most = 2_000_000 if prec == "f32" else 250_000
        ppc = max(1, min(ppc, most // (width * ny)))
        return dict(kind=kind, nx=nx, ny=ny, slab0=nx // 2, slab1=nx // 2 + width, ppc=ppc,
                    a0=round(rng.uniform(10.0, 30.0), 2), prec=prec, sort=16, steps=16, particles=prec == "f64")
    if kind == "qed":
        dim = rng.choice([2, 2, 3])
        n = [_log_int(rng, 100, 512), _log_int(rng, 100, 256), 1] if dim == 2 else [_log_int(rng, 24, 56) for _ in range(3)]
        return dict(kind=kind, dim=dim, nx=n[0], ny=n[1], nz=n[2],
                    electrons=_log_int(rng, 50_000, 1_000_000) if dim == 2 else _log_int(rng, 20_000, 200_000),
                    gamma0=round(rng.uniform(1200.0, 2400.0), 1), B0=round(rng.uniform(150.0, 250.0), 1),
                    mode=rng.choice(["table", "surrogate"]), sort=8, steps=rng.choice([4, 8]))
    if kind == "cascade":
        return dict(kind=kind, replicas=_log_int(rng, 200, 2000), gamma0=round(rng.uniform(500.0, 1500.0), 1),
                    b=round(rng.uniform(0.002, 0.009), 5), steps=rng.randint(100, 350))
    return dict(kind=kind, process=rng.choice([0, 1]), batch=128 * rng.randint(16, 128), iterations=rng.randint(20, 100))


# ---------------------------------------------------------------------------
# inputs (on the GPU, from the seed alone)
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(n, g):
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda")


def _randn(n, g):
    return torch.randn(n, generator=g, dtype=torch.float64, device="cuda")


def _dims(case):
    return case.get("dim", 2), (case["nx"], case["ny"], case.get("nz", 1))


def _set_up(case, seed):
    """Grid, species [(q, m, w, x[3], u[3])], initial fields, laser, background charge."""
    g = _gen(seed)
    dim, n = _dims(case)
    bc = (pic.PERIODIC,) * 3
    fields, laser, rho_bg = {}, None, 0.0
    if case["kind"] == "plasma":
        dx = (case["dx"],) * 3
        dt = 0.95 * case["dx"] / math.sqrt(dim)
        cells = n[0] * n[1] * n[2]
        N = cells * case["ppc"]
        if case["amp"] > 0.0:  # the cold oscillation: a quiet start, the seed moves its phase
            x0 = (torch.arange(N, device="cuda", dtype=torch.float64) + 0.5) * (n[0] * dx[0] / N)
            ph = TWO_PI * float(_rand(1, g))
            x = [x0, None, None]
            u = [case["amp"] * torch.sin(TWO_PI * x0 / (n[0] * dx[0]) + ph), torch.zeros_like(x0), torch.zeros_like(x0)]
        else:
            s = math.sqrt(case["T_keV"] / MEC2_KEV)
            x = [_rand(N, g) * (n[d] * dx[d]) if d < dim else None for d in range(3)]
            u = [_randn(N, g) * s for _ in range(3)]
        rho_bg = 1.0
        return dim, n, dx, dt, bc, [(-1.0, 1.0, 1.0 / case["ppc"], x, u)], fields, laser, rho_bg
    # foil: lambda = 1 um, 64 cells per wavelength, density 10 n_c, 1 keV
    dx = (TWO_PI / 64.0,) * 3
    dt = 0.95 * dx[0] / math.sqrt(2.0)
    bc = (pic.ABSORB, pic.PERIODIC, pic.PERIODIC)
    s0, s1 = case["slab0"], case["slab1"]
    N = (s1 - s0) * n[1] * case["ppc"]
    species = []
    for q, m in ((-1.0, 1.0), (1.0, M_PROTON)):
        x = [(s0 + (s1 - s0) * _rand(N, g)) * dx[0], _rand(N, g) * (n[1] * dx[1]), None]
        s = math.sqrt(1.0 / MEC2_KEV / m)
        species.append((q, m, 10.0 / case["ppc"], x, [_randn(N, g) * s for _ in range(3)]))
    # a 30 fs, 3 um pulse whose centre is 0.8 FWHM before the slab at t = 0
    # (or as far before it as the box has room), in the box and still entering
    omega_L = TWO_PI * 2.99792458e8 / 1.0e-6
    fwhm = min(30e-15 * omega_L, s0 * dx[0])
    xc = s0 * dx[0] - 0.8 * fwhm
    # (circular, so that the laser drives every component)
    laser = dict(a0=case["a0"], waist=3.0 * TWO_PI, fwhm=fwhm, t_peak=-xc, x_focus=s0 * dx[0], yc=0.5 * n[1] * dx[1],
                 pol=1)

    def pulse(i_off, j_off, wave):
        X = (torch.arange(n[0] + 1, device="cuda", dtype=torch.float64) + i_off) * dx[0]
        Y = (torch.arange(n[1], device="cuda", dtype=torch.float64) + j_off) * dx[1]
        tau = (xc - X)[None, None, :]
        f = torch.exp(-2.0 * math.log(2.0) * (tau / fwhm) ** 2) * wave(tau) * (X < s0 * dx[0])
        return case["a0"] * f * torch.exp(-(((Y - laser["yc"]) / laser["waist"]) ** 2))[None, :, None]

    fields = {pic.EY: pulse(0.0, 0.5, torch.sin), pic.EZ: pulse(0.0, 0.0, torch.cos),
              pic.BY: -pulse(0.5, 0.0, torch.cos), pic.BZ: pulse(0.5, 0.5, torch.sin)}
    for c in (pic.BY, pic.BZ):
        fields[c][..., -1] = 0.0  # beyond the last half node
    return dim, n, dx, dt, bc, species, fields, laser, rho_bg


def _host(t):
    return None if t is None else t.cpu().numpy()


class _Array:
    """A borrowed device array for torch (the CUDA array interface).  torch
    keeps this object as long as a tensor looks at the array, and this object
    keeps the simulation that owns the memory."""

    def __init__(self, sim, v, shape):
        self.sim = sim
        b = v["elem_bytes"]
        self.__cuda_array_interface__ = {
            "shape": shape, "typestr": "<f%d" % b, "data": (v["data"] + b * v["origin"], False), "version": 3,
            "strides": tuple(b * s for s in (v["stride"][2], v["stride"][1], v["stride"][0]))}


def _views(sim):
    return {name: torch.as_tensor(_Array(sim, sim.pic_field_device(c), sim.box()), device="cuda")
            for c, name in enumerate(COMPS)}


_NETS = {}


def _nets(sim):
    """The surrogate networks: trained once per process, as a program that runs many simulations does."""
    for p in (pic.QED_EMISSION, pic.QED_PAIR):
        if p not in _NETS:
            sim.pic_mlp_train(p, iterations=12000, seed=7)
            _NETS[p] = sim.pic_mlp_get(p)
        P, info = _NETS[p]
        sim.pic_mlp_set(p, P, info["chi_min"], info["chi_max"], info["mu"], info["sd"])


def prepare(case, seed):
    if case["kind"] == "train":
        sim = pic.pic_create(1, (16,), (1.0,), 0.1, [(-1.0, 1.0, 1.0, 16)])
        sim.pic_set_qed()
        return {"case": case, "sim": sim, "seed": seed}
    if case["kind"] == "cascade":
        w = W.cascade(case["gamma0"], case["b"], replicas=case["replicas"], steps=case["steps"], seed=seed)
        return {"case": case, "w": w, "seed": seed}
    if case["kind"] == "qed":
        # electrons of the collision's energy and spread, in random
        # directions, across a uniform B_z of half the pulse's peak force; they
        # cool until they emit no photon that is kept, and the photons stay
        dim, n = _dims(case)
        dx = (TWO_PI / 32.0,) * 3
        dt = 0.95 * dx[0] / math.sqrt(dim)
        N = case["electrons"]
        g = _gen(seed)
        gam = case["gamma0"] * (1.0 + 0.01 * _randn(N, g))
        um = torch.sqrt(gam * gam - 1.0)
        x = [_rand(N, g) * (n[d] * dx[d]) if d < dim else None for d in range(3)]
        ph, ct = TWO_PI * _rand(N, g), (2.0 * _rand(N, g) - 1.0) if dim == 3 else torch.zeros(N, device="cuda", dtype=torch.float64)
        st = torch.sqrt(1.0 - ct * ct)
        w = 1e-12  # weightless, as in the field sample: the events do not hang on the order of atomic sums
        # room for every photon above 10 MeV that the electrons can emit until they are slow
        spec = [(-1.0, 1.0, w, 3 * N, pic.KIND_MASSIVE, 1), (1.0, 1.0, w, 2 * N, pic.KIND_MASSIVE, 1),
                (0.0, 0.0, w, 48 * N, pic.KIND_PHOTON, 0)]
        sim = pic.pic_create(dim, n, dx, dt, spec, sort_interval=case["sort"],
                             tile=(16, 16, 1) if dim == 2 else (4, 4, 4), seed=seed)
        mode = pic.QED_SURROGATE if case["mode"] == "surrogate" else pic.QED_TABLE
        sim.pic_set_qed(photon_sp=2, electron_sp=0, positron_sp=1, lambda_r_m=1e-6, photon_emin=20.0, mode=mode)
        if mode == pic.QED_SURROGATE:
            _nets(sim)
        sim.pic_set_field(pic.BZ, case["B0"])
        sim.pic_load_particles(0, *[_host(v) for v in x], _host(um * st * torch.cos(ph)), _host(um * st * torch.sin(ph)),
                               _host(um * ct))
        return {"case": case, "sim": sim, "fields": _views(sim)}
    dim, n, dx, dt, bc, species, fields, laser, rho_bg = _set_up(case, seed)
    tile = {1: (16, 1, 1), 2: (16, 16, 1), 3: (4, 4, 4)}[dim]
    sim = pic.pic_create(dim, n, dx, dt, [(q, m, w, len(u[0])) for q, m, w, x, u in species], bc=bc,
                         precision=PREC[case["prec"]], sort_interval=case["sort"], tile=tile, rho_bg=rho_bg,
                         order=case.get("order", 2))
    if laser:
        sim.pic_set_laser(**laser)
    for c, v in fields.items():
        sim.pic_set_field(c, _host(v))
    for i, (q, m, w, x, u) in enumerate(species):
        sim.pic_load_particles(i, *[_host(v) for v in x], *[_host(v) for v in u])
    return {"case": case, "sim": sim, "fields": _views(sim)}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _energies(d):
    return {"U_E": d["U_E"], "U_B": d["U_B"], "U_kin": d["U_kin"]}


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        rep = state["sim"].pic_mlp_train(case["process"], iterations=case["iterations"], batch=case["batch"],
                                         seed=state["seed"])
        params, _ = state["sim"].pic_mlp_get(case["process"])
        return {"params": params, "loss": rep["loss"], "rms_err_s": rep["rms_err_s"]}
    if case["kind"] == "cascade":
        w = state["w"]
        with pic.from_workload(w, seed=state["seed"]) as sim:
            sim.pic_set_qed(method=2, **w.qed)
            sim.pic_set_field(pic.BZ, w.notes["B0"])
            sim.pic_step(w.steps)
            parts = [sim.pic_get_particles(i) for i in range(3)]
        # records of one size whatever the number of events: the momenta, then zeros
        rec = {s.name: np.zeros((3, s.capacity), np.float32) for s in w.species}
        for s, p in zip(w.species, parts):
            for r, k in zip(rec[s.name], ("ux", "uy", "uz")):
                r[: len(p[k])] = p[k]
        return rec
    sim = state["sim"]
    sim.pic_step(case["steps"])
    out = {"fields": state["fields"]}
    if case["kind"] == "qed" or case.get("log"):
        out["energies"] = _energies(sim.pic_diagnostics())
    if case.get("dump"):
        out["snapshot"] = {name: sim.pic_fields(c).astype(np.float32) for c, name in enumerate(COMPS + ("rho",))}
    if case.get("particles"):
        out["particles"] = [{k: p[k] for k in ("x", "y", "ux", "uy", "uz")}
                            for p in (sim.pic_get_particles(i) for i in range(sim.nsp))]
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "train":  # forward, and twice that backward, of 2-64-64-64-2 on every row
        macs = 2 * 64 + 2 * 64 * 64 + 64 * 2
        return {"bytes": 4.0 * 8642 * 8 * case["iterations"], "flops": 6.0 * macs * case["batch"] * case["iterations"]}
    if case["kind"] == "cascade":  # some 40 photons a replica on average over the run; each moves every step (1D, FP32)
        live = 40.0 * case["replicas"]
        return {"bytes": live * case["steps"] * (2 * 20 + 24), "flops": live * case["steps"] * 300.0}
    dim, n = _dims(case)
    cells = float(n[0] * n[1] * n[2])
    per = 350.0 if dim == 2 else (800.0 if dim == 3 else 150.0)
    if case["kind"] == "qed":
        # leptons: cell, offsets, u, optical depth in and out, identity in;
        # photons (some 20 an electron over the run): the same, k only in
        N = case["electrons"]
        lep, pho = 2.0 * (4 + 4 * dim + 12 + 8) + 8, 2.0 * (4 + 4 * dim + 8) + 12
        return {"bytes": case["steps"] * (N * (lep + 20 * pho) + cells * 9 * 4 * 2),
                "flops": case["steps"] * N * (per + 100.0 + 20 * 0.6 * per)}
    r = 8.0 if case["prec"] == "f64" else 4.0
    if case["kind"] == "foil":
        N = 2.0 * (case["slab1"] - case["slab0"]) * case["ny"] * case["ppc"]
    else:
        N = cells * case["ppc"]
    state = r * (dim + 3) + 4.0
    if case.get("order", 2) == 4:
        per *= 2.5
    out = (N * 40.0 if case.get("particles") else 0.0) + (cells * 10 * 8.0 if case.get("dump") else 0.0)
    return {"bytes": case["steps"] * (2.0 * N * state + 2.0 * cells * 9 * r) + out, "flops": case["steps"] * N * per}


# ---------------------------------------------------------------------------
# the same pass in 64 bits (plain torch)
# ---------------------------------------------------------------------------
class _Ref:
    """The split PIC step in FP64 torch: periodic axes are rolled; an absorbing
    x axis is padded by 4 and carries the first-order Mur condition on the
    scattered tangential B (y periodic there).  Arrays are [z, y, x]."""

    def __init__(self, dim, n, dx, dt, bc, order, laser):
        self.dim, self.n, self.dx, self.dt, self.order, self.laser = dim, n, dx, dt, order, laser
        self.absorb = bc[0] == pic.ABSORB
        self.G = 4 if self.absorb else 0
        self.shape = (n[2], n[1], n[0] + 1 + 2 * self.G if self.absorb else n[0])
        self.F = [torch.zeros(self.shape, dtype=torch.float64, device="cuda") for _ in range(9)]
        self.t = 0.0
        i = torch.arange(self.shape[2], device="cuda") - self.G
        self.node = (i >= 0) & (i <= n[0]) if self.absorb else torch.ones_like(i, dtype=torch.bool)
        self.half = (i >= 0) & (i <= n[0] - 1) if self.absorb else self.node

    def box(self, a):
        return a[..., self.G:self.G + self.n[0] + 1] if self.absorb else a

    def d(self, a, axis, side):  # difference over one cell: side +1 forward, -1 backward
        if axis >= self.dim:
            return 0.0
        b = torch.roll(a, -side, dims=2 - axis)
        return (b - a if side > 0 else a - b) / self.dx[axis]

    def update_E(self, h):
        E, B, J, d = self.F[:3], self.F[3:6], self.F[6:], self.d
        curl = [d(B[2], 1, -1) - d(B[1], 2, -1), d(B[0], 2, -1) - d(B[2], 0, -1), d(B[1], 0, -1) - d(B[0], 1, -1)]
        for c in range(3):
            E[c] += h * (curl[c] - J[c]) * (self.half if c == 0 else self.node)

    def incident(self, comp, tau):  # the laser's B_z = E_y or B_y = -E_z at x = 0 and time tau (circular)
        L = self.laser
        if not L:
            return 0.0
        Y = (torch.arange(self.n[1], device="cuda", dtype=torch.float64) + (0.5 if comp == 2 else 0.0)) * self.dx[1]
        xr, xi = 0.5 * L["waist"] ** 2, -L["x_focus"]
        wx = L["waist"] * math.sqrt(1.0 + (xi / xr) ** 2)
        r2 = (Y - L["yc"]) ** 2
        ph = -0.5 * r2 * xi / (xi * xi + xr * xr) + 0.5 * math.atan(xi / xr)
        amp = L["a0"] * math.sqrt(L["waist"] / wx) * torch.exp(-r2 / (wx * wx))
        a = (tau - L["t_peak"]) / L["fwhm"]
        wave = torch.sin if comp == 2 else (lambda v: -torch.cos(v))
        return (amp * math.exp(-2.0 * math.log(2.0) * a * a) * wave(tau - L["t_peak"] + ph))[None, :]

    def update_B(self, h, t_new):
        E, B, d = self.F[:3], self.F[3:6], self.d
        curl = [d(E[2], 1, 1) - d(E[1], 2, 1), d(E[0], 2, 1) - d(E[2], 0, 1), d(E[1], 0, 1) - d(E[0], 1, 1)]
        old = [b.clone() for b in B]
        for c in range(3):
            B[c] -= h * curl[c] * (self.node if c == 0 else self.half)
        if not self.absorb:
            return
        a, hx = h / self.dx[0], 0.5 * self.dx[0]
        c1 = (a - 1.0) / (a + 1.0)
        for c in (1, 2):
            for ghost, inner, inc in ((self.G - 1, self.G, True), (self.G + self.n[0], self.G + self.n[0] - 1, False)):
                f = (lambda tau: self.incident(c, tau)) if inc else (lambda tau: 0.0)
                B[c][..., ghost] = f(t_new + hx) + (old[c][..., inner] - f(t_new - h - hx)) + c1 * (
                    (B[c][..., inner] - f(t_new - hx)) - (B[c][..., ghost] - f(t_new - h + hx)))

    def weights(self, X, stag):  # nearest node and the ORDER + 1 weights about it
        ic = torch.floor(X) if stag else torch.floor(X + 0.5)
        e = X - ic - (0.5 if stag else 0.0)
        if self.order == 2:
            w = [0.5 * (0.5 - e) ** 2, 0.75 - e * e, 0.5 * (0.5 + e) ** 2]
        else:
            e2 = e * e
            w = [(1 - 2 * e) ** 4 / 384, (19 - 44 * e + 24 * e2 + 16 * e2 * e - 16 * e2 * e2) / 96,
                 115 / 192 - 0.625 * e2 + 0.25 * e2 * e2, (19 + 44 * e + 24 * e2 - 16 * e2 * e - 16 * e2 * e2) / 96,
                 (1 + 2 * e) ** 4 / 384]
        return ic.to(torch.int64), w

    def index(self, d, i):
        return i + self.G if d == 0 and self.absorb else i % self.n[d]

    def at(self, idx):  # flat index of (x, y, z) indices (absent axes at 0)
        o = idx[0]
        if self.dim > 1:
            o = o + self.shape[2] * idx[1]
        if self.dim > 2:
            o = o + self.shape[2] * self.shape[1] * idx[2]
        return o

    def gather(self, X):
        H, P = self.order // 2, self.order + 1
        sh = [[self.weights(X[d], s) for s in (0, 1)] for d in range(self.dim)]
        ix = [[[self.index(d, sh[d][s][0] + (k - H)) for k in range(P)] for s in (0, 1)] for d in range(self.dim)]
        out = []
        for c in range(6):
            st = [int((c < 3) == (d == c % 3)) for d in range(3)]
            F, acc = self.F[c].reshape(-1), 0.0
            for k in range(P if self.dim > 2 else 1):
                for j in range(P if self.dim > 1 else 1):
                    for i in range(P):
                        m = (i, j, k)
                        w = 1.0
                        for d in range(self.dim):
                            w = w * sh[d][st[d]][1][m[d]]
                        acc = acc + w * F[self.at([ix[d][st[d]][m[d]] for d in range(self.dim)])]
            out.append(acc)
        return out

    def deposit(self, X0, X1, v, qw):  # Esirkepov on the straight path X0 -> X1
        H, P, WN = self.order // 2, self.order + 1, self.order + 3
        S, D, ix = [], [], []
        for d in range(self.dim):
            i0, w0 = self.weights(X0[d], 0)
            i1, w1 = self.weights(X1[d], 0)
            z = torch.zeros_like(X0[d])
            s0 = [z] + w0 + [z]
            sft = i1 - i0
            pad = [z, z] + w1 + [z, z]
            s1 = [torch.where(sft == 0, pad[k + 1], torch.where(sft > 0, pad[k], pad[k + 2])) for k in range(WN)]
            S.append(s0)
            D.append([b - a for a, b in zip(s0, s1)])
            ix.append([self.index(d, i0 + (k - H - 1)) for k in range(WN)])
        J = [a.reshape(-1) for a in self.F[6:]]
        for c in range(3):
            oth = [d for d in range(self.dim) if d != c]

            def mean(m):  # time average of the product of the other axes' shapes
                if len(oth) == 1:
                    a = oth[0]
                    return S[a][m[0]] + 0.5 * D[a][m[0]]
                if len(oth) == 0:
                    return 1.0
                (a, b), (i, j) = oth, m
                return S[a][i] * S[b][j] + 0.5 * (D[a][i] * S[b][j] + S[a][i] * D[b][j]) + D[a][i] * D[b][j] / 3.0

            grid = [range(WN)] * len(oth)
            for m in [()] if not grid else [(i,) for i in grid[0]] if len(grid) == 1 else [(i, j) for i in grid[0] for j in grid[1]]:
                t = mean(m)
                idx = [None] * self.dim
                for d, i in zip(oth, m):
                    idx[d] = ix[d][i]
                if c < self.dim:
                    acc = 0.0
                    for k in range(WN - 1):
                        acc = acc - qw * self.dx[c] / self.dt * D[c][k] * t
                        idx[c] = ix[c][k]
                        J[c].index_add_(0, self.at(idx), acc)
                else:
                    J[c].index_add_(0, self.at(idx), qw * v[c] * t)

    def step(self, species, chunk=1 << 21):
        h = 0.5 * self.dt
        self.update_E(h)
        self.update_B(h, self.t + h)
        for a in self.F[6:]:
            a.zero_()
        for q, m, w, x, u in species:
            for s in range(0, len(u[0]), chunk):
                e = slice(s, s + chunk)
                U = [v[e] for v in u]
                ig = 1.0 / torch.sqrt(1.0 + U[0] ** 2 + U[1] ** 2 + U[2] ** 2)
                Xh = [x[d][e] + h * U[d] * ig for d in range(self.dim)]
                k = 0.5 * self.dt * q / m
                f = [k * v for v in self.gather([a / b for a, b in zip(Xh, self.dx)])]
                U = [a + b for a, b in zip(U, f[:3])]
                ig = 1.0 / torch.sqrt(1.0 + U[0] ** 2 + U[1] ** 2 + U[2] ** 2)
                t = [b * ig for b in f[3:]]
                s2 = 2.0 / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
                up = [U[a] + U[(a + 1) % 3] * t[(a + 2) % 3] - U[(a + 2) % 3] * t[(a + 1) % 3] for a in range(3)]
                U = [U[a] + s2 * (up[(a + 1) % 3] * t[(a + 2) % 3] - up[(a + 2) % 3] * t[(a + 1) % 3]) + f[a] for a in range(3)]
                ig = 1.0 / torch.sqrt(1.0 + U[0] ** 2 + U[1] ** 2 + U[2] ** 2)
                v = [a * ig for a in U]
                X1 = [Xh[d] + h * v[d] for d in range(self.dim)]
                X2 = [X1[d] + h * v[d] for d in range(self.dim)]
                self.deposit([a / b for a, b in zip(Xh, self.dx)], [a / b for a, b in zip(X2, self.dx)], v, q * w)
                for d in range(self.dim):
                    L = self.n[d] * self.dx[d]
                    x[d][e] = X1[d] if d == 0 and self.absorb else torch.where(X1[d] < 0, X1[d] + L, torch.where(X1[d] >= L, X1[d] - L, X1[d]))
                for a in range(3):
                    u[a][e] = U[a]
        self.update_B(h, self.t + self.dt)
        self.update_E(h)
        self.t += self.dt

    def rho(self, species):  # the charge density averaged over x -/+ (dt/2) v
        P, H = self.order + 1, self.order // 2
        out = torch.zeros(self.shape, dtype=torch.float64, device="cuda").reshape(-1)
        for q, m, w, x, u in species:
            ig = 1.0 / torch.sqrt(1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
            for side in (-0.5, 0.5):
                sh = [self.weights((x[d] + side * self.dt * u[d] * ig) / self.dx[d], 0) for d in range(self.dim)]
                for k in range(P if self.dim > 2 else 1):
                    for j in range(P if self.dim > 1 else 1):
                        for i in range(P):
                            mm, t = (i, j, k), 0.5 * q * w
                            for d in range(self.dim):
                                t = t * sh[d][1][mm[d]]
                            out.index_add_(0, self.at([self.index(d, sh[d][0] + (mm[d] - H)) for d in range(self.dim)]), t)
        return out.reshape(self.shape)


def exact(case, seed):
    if case["kind"] not in ("plasma", "foil"):
        return None  # Monte Carlo decisions and a training run have no 64-bit value of their own
    dim, n, dx, dt, bc, species, fields, laser, _ = _set_up(case, seed)
    if max(len(s[4][0]) for s in species) * case["steps"] > 100_000_000:
        return None
    ref = _Ref(dim, n, dx, dt, bc, case.get("order", 2), laser)
    for c, v in fields.items():
        ref.box(ref.F[c]).copy_(v)
    if case.get("particles"):  # returned in the order of the sort before the first step: by 16 x 16 tile, then by cell
        for i, (q, m, w, x, u) in enumerate(species):
            cx, cy = (torch.floor(x[d] / dx[d]).to(torch.int64) for d in (0, 1))
            key = (cy // 16 * ((n[0] + 15) // 16) + cx // 16) * 256 + cy % 16 * 16 + cx % 16
            p = torch.sort(key, stable=True).indices
            species[i] = (q, m, w, [None if a is None else a[p] for a in x], [a[p] for a in u])
    for _ in range(case["steps"]):
        ref.step(species)
    out = {"fields": {name: ref.box(a) for name, a in zip(COMPS, ref.F)}}
    dV = math.prod(dx[:dim])
    if case.get("log"):
        cut = slice(0, n[0])
        kin = []
        for q, m, w, x, u in species:
            uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
            kin.append((uu / (torch.sqrt(1.0 + uu) + 1.0)).sum() * (w * m * dV))
        en = [0.5 * dV * sum((ref.box(ref.F[3 * k + c])[..., cut] ** 2).sum() for c in range(3)) for k in (0, 1)]
        out["energies"] = {"U_E": en[0], "U_B": en[1], "U_kin": kin}
    if case.get("dump"):
        out["snapshot"] = dict(out["fields"], rho=ref.box(ref.rho(species)))
    if case.get("particles"):
        out["particles"] = [{"x": x[0], "y": x[1], "ux": u[0], "uy": u[1], "uz": u[2]} for q, m, w, x, u in species]
    return out
