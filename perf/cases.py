"""Performance cases of the framework: what its users have it do, through its public entry points.

Kinds of case (every size is a power of two per side, as the library requires):

  steps     a run advances by `steps` COLA steps: the particle state is restored (as from a
            checkpoint), cola_step is called once, and the new state is read back on the device
  batch     an ensemble of same-shape runs with mixed models advances together, through a
            Batch or (loop) tick by tick through step_many as a serving loop does
  job       a whole run from its configuration: context, initial conditions, every step,
            P(k), displacements and velocities
  spectrum  analysis of a state: P(k) to the host and a snapshot on the device
  transform the 3-D real transform forward and back, on device arrays
  mesh      CIC deposit of caller positions and the force from a caller density

Inputs are made from the seed with torch: Gaussian 2LPT potentials, and particle states on the
LPT trajectory at the step they start from, with a share of the Lagrangian blocks collapsed into
clumps about a mesh cell wide (the clustering of late steps).  `exact` evaluates the same method
in double precision with plain numpy and torch.
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1703_00879_gb300 as pkg

LCDM, FOFR, NDGP = pkg.COLA_LCDM, pkg.COLA_FOFR, pkg.COLA_NDGP
OM, OB, H, NS, SIGMA8 = 0.3, 0.05, 0.7, 0.97, 0.8
Z_INI, NK, C_LIGHT = 19.0, 1024, 2997.92458
F64 = torch.float64


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, Np=64, Nmesh=128, Lbox=128.0, nsteps=30, start=15, steps=4, model=LCDM, fR0=0.0,
             rcH0=0.0, screening=0, seed_precision=0, lpt_fast=False, sims=1, loop=False, npos=0, nbins=0)
    c.update(kw)
    return c


def listed():
    fr = dict(model=FOFR, fR0=1e-5, screening=1)
    dgp = dict(model=NDGP, rcH0=1.0, screening=1)
    return [
        # the small parity workload, run whole in one call: launches and latency are all of it
        _case("steps_32p_32m_fofr", "steps", Np=32, Nmesh=32, Lbox=64.0, nsteps=10, start=0, steps=10, **fr),
        # one ensemble member stepped alone (the one-at-a-time rate)
        _case("steps_64p_128m_ndgp", "steps", nsteps=20, start=8, steps=8, model=NDGP, rcH0=5.0, screening=1),
        # the ensemble: 256 members, the six models of the ensemble in turn
        _case("batch_256x64p_128m", "batch", sims=256, nsteps=20, start=8, steps=4),
        # the bench's model and resolution on a sub-box
        _case("steps_128p_256m_ndgp", "steps", Np=128, Nmesh=256, Lbox=256.0, start=15, steps=6, **dgp),
        # the main f(R) workload, late steps
        _case("steps_256p_512m_fofr", "steps", Np=256, Nmesh=512, Lbox=512.0, start=20, steps=4, **fr),
        # the bench workload
        _case("steps_512p_1024m_ndgp", "steps", Np=512, Nmesh=1024, Lbox=1024.0, start=12, steps=4, **dgp),
        # the LCDM twin of a boost measurement, scale-independent path, mesh as coarse as the lattice
        _case("steps_256p_256m_lcdm_fast", "steps", Np=256, Nmesh=256, Lbox=512.0, start=10, steps=5, lpt_fast=True),
        # half-precision seeds and fields, unscreened f(R), one step per call
        _case("steps_256p_512m_fofr_fp16", "steps", Np=256, Nmesh=512, Lbox=512.0, start=2, steps=1, model=FOFR,
              fR0=1e-6, screening=0, seed_precision=2),
        # a served request from configuration to P(k)
        _case("job_128p_256m_ndgp", "job", Np=128, Nmesh=256, Lbox=256.0, nsteps=10, **dgp),
        # analysis of a snapshot
        _case("spectrum_256p_512m", "spectrum", Np=256, Nmesh=512, Lbox=512.0, start=20, nbins=255, **fr),
        # the transforms on their own
        _case("transform_512m", "transform", Np=32, Nmesh=512, Lbox=512.0),
        # stage entry points on caller data, a number of positions that fits no tile
        _case("mesh_256m_fofr", "mesh", Np=128, Nmesh=256, Lbox=256.0, npos=2000003, **fr),
    ]


def draw(rng):
    kind = rng.choice(["steps"] * 8 + ["batch"] * 2 + ["job", "spectrum", "transform", "mesh"])
    model = rng.choice([LCDM, FOFR, FOFR, NDGP, NDGP])
    c = _case("", kind, model=model)
    del c["name"]
    if model == FOFR:
        c["fR0"] = 10.0 ** rng.uniform(-6.0, -4.0)
    elif model == NDGP:
        c["rcH0"] = rng.uniform(0.5, 5.0)
    c["screening"] = int(model != LCDM and rng.random() < 0.8)
    top = {"steps": 9, "batch": 6, "job": 8, "spectrum": 8, "transform": 5, "mesh": 8}[kind]
    c["Np"] = 1 << rng.randint(5, top)
    c["Nmesh"] = max(32, c["Np"] * rng.choice([1, 2, 2, 2]))
    if rng.random() < 0.1:  # a mesh coarser than the lattice
        c["Nmesh"] = max(32, c["Np"] // 2)
    if kind == "transform":
        c["Np"], c["Nmesh"] = 32, 1 << rng.randint(5, 10)
    c["Lbox"] = c["Np"] * rng.uniform(1.0, 3.0)
    c["nsteps"] = rng.randint(10, 30)
    c["start"] = rng.randint(0, c["nsteps"] - 4)
    c["steps"] = rng.randint(1, 4)
    if kind == "steps":
        if rng.random() < 0.15:
            c["seed_precision"] = rng.choice([1, 2])
            c["start"] = rng.randint(0, 2)
        elif model != FOFR and rng.random() < 0.25:
            c["lpt_fast"] = True
    elif kind == "batch":
        c["sims"] = int(round(2.0 ** rng.uniform(1.0, 9.0 - 3.0 * (c["Np"] == 64) * (c["Nmesh"] == 128))))
        c["loop"] = rng.random() < 0.4
    elif kind == "job":
        c["nsteps"] = rng.randint(10, 14)
    elif kind == "spectrum":
        c["nbins"] = rng.randint(c["Nmesh"] // 4, c["Nmesh"] // 2 - 1)
    elif kind == "mesh":
        c["npos"] = int(10.0 ** rng.uniform(3.0, 7.0))
    return c


# ------------------------------------------------------------------ configuration records

def _models(case):
    """The model of every simulation of a case (ensembles cycle through six)."""
    if case["kind"] == "batch":
        six = [(LCDM, 0.0, 0.0, 0)] + [(FOFR, f, 0.0, 1) for f in (1e-6, 1e-5, 1e-4)] + [(NDGP, 0.0, r, 1) for r in (1.0, 5.0)]
        return [six[i % 6] for i in range(case["sims"])]
    return [(case["model"], case["fR0"], case["rcH0"], case["screening"])] * case["sims"]


def _run_record(case, model, seed):
    kind, fR0, rcH0, scr = model
    return SimpleNamespace(
        Np=case["Np"], Nmesh=case["Nmesh"], Lbox=case["Lbox"], nsteps=case["nsteps"], z_ini=Z_INI, z_final=0.0, seed=seed,
        nk_table=NK, cosmo=SimpleNamespace(Omega_m=OM, Omega_b=OB, h=H, n_s=NS, sigma8=SIGMA8),
        model=SimpleNamespace(kind=kind, fR0=fR0, rcH0=rcH0, screening=scr, R_smooth=1.0, scale_dependent=1))


# ------------------------------------------------------------------ background and growth (double precision)

def _E(a):
    return math.sqrt(OM / a**3 + 1.0 - OM)


def _fr_x(a):
    return (OM / a**3 + 4.0 * (1.0 - OM)) / (OM + 4.0 * (1.0 - OM))


def _fr_m2(a, fR0):
    return (OM + 4.0 * (1.0 - OM)) / (2.0 * fR0) * _fr_x(a) ** 3 / C_LIGHT**2


def _dgp_beta(a, rcH0):
    return 1.0 + 2.0 * rcH0 * _E(a) * (1.0 - 0.5 * OM / (a**3 * _E(a) ** 2))


def _mu_gamma(model, k, a):
    """mu(k, a) and gamma_2 at the orthogonal triangle (Sec. 5.1, Sec. 5.2)."""
    kind, fR0, rcH0, _ = model
    if kind == FOFR:
        ol4 = 4.0 * (1.0 - OM)
        x = (k * C_LIGHT / a) ** 2
        m = (OM / a**3 + ol4) ** 3 / (2.0 * fR0 * (OM + ol4) ** 2)
        g = -9.0 * OM**2 / (48.0 * a**6 * fR0**2) * x / _E(a) ** 2 * (OM / a**3 + ol4) ** 5 / (OM + ol4) ** 4
        return 1.0 + k**2 / (3.0 * (k**2 + a * a * _fr_m2(a, fR0))), g / ((x + m) * (0.5 * x + m) ** 2)
    if kind == NDGP:
        b = _dgp_beta(a, rcH0)
        return np.full_like(k, 1.0 + 1.0 / (3.0 * b)), np.full_like(k, -(rcH0 * OM / _E(a)) ** 2 / (6.0 * b**3 * a**6))
    return np.ones_like(k), np.zeros_like(k)


def _growth(model, a_nodes, k):
    """Rows (D1, D1', D1'', D2, D2', D2'') over k at every a node, by RK4 in ln a (Sec. 4.1, Eq. fofrapprox)."""
    def second(a, y):
        mu, g2 = _mu_gamma(model, k, a)
        kap = 1.5 * OM * a
        return kap * mu * y[0], kap * mu * (y[2] - y[0] ** 2) - 2.0 * a**4 * _E(a) ** 2 * g2 * y[0] ** 2

    def rhs(t, y):
        a = math.exp(t)
        d1, d2 = second(a, y)
        return np.stack([y[1], d1, y[3], d2]) / (a * a * _E(a))

    a0 = a_nodes[0]
    one = np.ones_like(k)
    w = a0 * a0 * _E(a0)
    y, rows = np.stack([one, w * one, -3.0 / 7.0 * one, -6.0 / 7.0 * w * one]), []
    for i, a in enumerate(a_nodes):
        if i:
            t0, t1 = math.log(a_nodes[i - 1]), math.log(a)
            n = max(4, int(math.ceil((t1 - t0) / 0.005)))
            h = (t1 - t0) / n
            for j in range(n):
                t = t0 + j * h
                k1 = rhs(t, y)
                k2 = rhs(t + 0.5 * h, y + 0.5 * h * k1)
                k3 = rhs(t + 0.5 * h, y + 0.5 * h * k2)
                k4 = rhs(t + h, y + h * k3)
                y = y + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        d1, d2 = second(a, y)
        rows.append(np.stack([y[0], y[1], d1, y[2], y[3], d2]))
    return rows


def _nodes(case):
    a0 = 1.0 / (1.0 + Z_INI)
    return [a0 + i * (1.0 - a0) / case["nsteps"] for i in range(case["nsteps"])] + [1.0]


def _table_k(case):
    lo, hi = math.log(math.pi / case["Lbox"]), math.log(1.01 * math.sqrt(3.0) * math.pi * case["Np"] / case["Lbox"])
    return lo, (hi - lo) / (NK - 1)


def _dtau(a, b):
    x, w = np.polynomial.legendre.leggauss(24)
    return float(sum(0.5 * (b - a) * wi / (u**3 * _E(u)) for u, wi in zip(0.5 * (b - a) * x + 0.5 * (a + b), w)))


# ------------------------------------------------------------------ inputs from the seed

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _grid(N, L):
    """(kx, ky, kz), k^2 and the derivative factors (zero on their own Nyquist plane) of a half spectrum [z][y][x]."""
    kf = 2.0 * math.pi / L
    full = torch.fft.fftfreq(N, 1.0 / N, dtype=F64, device="cuda") * kf
    half = torch.arange(N // 2 + 1, dtype=F64, device="cuda") * kf
    gf, gh = full.clone(), half.clone()
    gf[N // 2] = 0.0
    gh[N // 2] = 0.0
    sh = ((1, 1, -1), (1, -1, 1), (-1, 1, 1))
    k = [half.view(sh[0]), full.view(sh[1]), full.view(sh[2])]
    g = [gh.view(sh[0]), gf.view(sh[1]), gf.view(sh[2])]
    return k, k[0] ** 2 + k[1] ** 2 + k[2] ** 2, g


def _linear_shape(k):
    """CDM power spectrum shape k^ns T^2 with the BBKS transfer function (Bardeen et al. 1986)."""
    q = np.maximum(k, 1e-12) / (OM * H)
    t = np.log(1.0 + 2.34 * q) / (2.34 * q) * (1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
    return k**NS * t * t


@functools.lru_cache(maxsize=None)
def _lcdm_growth(a):
    """(D1, D2) of LCDM at a, D1 = 1 at a_ini."""
    r = _growth((LCDM, 0.0, 0.0, 0), [1.0 / (1.0 + Z_INI), a], np.ones(1))[1]
    return float(r[0][0]), float(r[3][0])


@functools.lru_cache(maxsize=None)
def _amplitude():
    k = np.exp(np.linspace(math.log(1e-4), math.log(50.0), 4000))
    x = 8.0 * k
    w = 3.0 * (np.sin(x) - x * np.cos(x)) / x**3
    var = np.sum(_linear_shape(k) * w * w * k**3) * math.log(50.0 / 1e-4) / 3999 / (2.0 * math.pi**2)
    return (SIGMA8 / _lcdm_growth(1.0)[0]) ** 2 / var


def _potentials(case, seed):
    """phi1(k), phi2(k) (complex64, dense half spectra) of a Gaussian field (Sec. 3.1, Sec. 3.2)."""
    N, L = case["Np"], case["Lbox"]
    k, k2, g = _grid(N, L)
    d = torch.fft.rfftn(torch.randn((N, N, N), generator=_generator(seed), dtype=F64, device="cuda"))
    amp = _amplitude() * N**3 / L**3
    kt = np.exp(np.linspace(math.log(0.5 * math.pi / L), math.log(2.0 * math.pi * N / L), 8192))
    root = torch.as_tensor(np.sqrt(amp * _linear_shape(kt)) / kt**2, device="cuda")
    u = ((0.5 * k2.clamp_min(1e-30).log() - math.log(kt[0])) / math.log(kt[1] / kt[0])).round().clamp(0, 8191).long()
    d *= root[u]
    del u
    d[0, 0, 0] = 0.0
    phi1 = d.to(torch.complex64)
    h = {(i, j): torch.fft.irfftn((-g[i] * g[j] if i != j else -k[i] * k[i]) * d, s=(N, N, N)) for i in range(3) for j in range(i, 3)}
    src = sum(h[i, i] * h[j, j] - h[i, j] ** 2 for i, j in ((0, 1), (0, 2), (1, 2)))
    del h
    k2[0, 0, 0] = 1.0
    phi2 = -torch.fft.rfftn(src) / k2
    phi2[0, 0, 0] = 0.0
    return phi1.contiguous(), phi2.to(torch.complex64).contiguous()  # rfftn may return permuted strides


def _state(case, seed, phi, n):
    """Displacement, residual velocity and residual acceleration [3, P] float32 at step n."""
    N, L, spacing = case["Np"], case["Lbox"], case["Lbox"] / case["Np"]
    a = _nodes(case)[n]
    gen = _generator(seed + 1)
    d1, d2 = _lcdm_growth(a)
    _, _, g = _grid(N, L)
    p1, p2 = (p.to(torch.complex128) for p in phi)
    s = torch.stack([torch.fft.irfftn(1j * gi * (d1 * p1 + d2 * p2), s=(N, N, N)) for gi in g])
    share = 0.0 if n == 0 else 0.4 * a
    B = N // 4
    blocks = (torch.rand((B, B, B), generator=gen, device="cuda") < share).repeat_interleave(4, 0).repeat_interleave(4, 1).repeat_interleave(4, 2)
    centre = torch.nn.functional.avg_pool3d(s, 4).repeat_interleave(4, 1).repeat_interleave(4, 2).repeat_interleave(4, 3)
    off = 1.5 * spacing - spacing * (torch.arange(N, device="cuda", dtype=F64) % 4)
    back = torch.stack([off.view(sh).expand(N, N, N) for sh in ((1, 1, -1), (1, -1, 1), (-1, 1, 1))])
    r = torch.randn((3, N, N, N), generator=gen, dtype=F64, device="cuda")
    s = torch.where(blocks, centre + back + 0.5 * spacing * r, s)
    sigma = torch.where(blocks, 3.0 * a, 0.0 if n == 0 else 0.2 * a)
    v = torch.randn((3, N, N, N), generator=gen, dtype=F64, device="cuda") * sigma
    acc = torch.randn((3, N, N, N), generator=gen, dtype=F64, device="cuda") * (0.1 * sigma + 0.01 * a)
    return [x.reshape(3, -1).float().contiguous() for x in (s, v, acc)]


def _seed_of(seed, i):
    return (int(seed) * 1000003 + 7919 * i) & 0x7FFFFFF


def _mesh_inputs(case, seed):
    N, L = case["Nmesh"], case["Lbox"]
    gen = _generator(seed)
    pos = (torch.rand((case["npos"], 3), generator=gen, device="cuda") * 1.2 - 0.1) * L
    centre = torch.rand((max(1, case["npos"] // 64), 3), generator=gen, device="cuda") * L
    pick = torch.randint(0, 3 * centre.shape[0], (case["npos"],), generator=gen, device="cuda")
    clump = pick < centre.shape[0]
    near = centre[pick.clamp_max(centre.shape[0] - 1)] + torch.randn((case["npos"], 3), generator=gen, device="cuda") * (L / N)
    pos = torch.where(clump[:, None], near, pos)
    mean = case["Np"] ** 3 / N**3
    rho = torch.exp(torch.randn((N, N, N), generator=gen, device="cuda") - 0.5) * mean
    return pos.contiguous(), rho


# ------------------------------------------------------------------ the cases

def prepare(case, seed):
    st = SimpleNamespace(case=case, kind=case["kind"])
    kind = case["kind"]
    if kind == "job":
        st.run = _run_record(case, _models(case)[0], int(seed))
        st.disp = torch.empty((3, case["Np"] ** 3), device="cuda")
        st.vel = torch.empty((case["Np"] ** 3, 3), device="cuda")
        return st
    st.sims, st.inp = [], []
    n = case["start"]
    single = kind in ("transform", "mesh")
    for i, m in enumerate(_models(case)):
        sim = pkg.Simulation(_run_record(case, m, i), seed_precision=case["seed_precision"], ic=False, lpt_fast=case["lpt_fast"])
        st.sims.append(sim)
        if not single:
            phi = _potentials(case, _seed_of(seed, i))
            pkg._check(pkg.lib().cola_ic_from_potentials(sim.ctx, phi[0].data_ptr(), phi[1].data_ptr(), pkg.COLA_DEVICE), sim.ctx)
            st.inp.append(_state(case, _seed_of(seed, i), phi, n))
            del phi
    N = case["Nmesh"]
    if kind == "transform":
        gen = _generator(seed)
        st.real = torch.randn((N, N, N), generator=gen, device="cuda")
        st.spec = torch.fft.rfftn(torch.randn((N, N, N), generator=gen, device="cuda")).contiguous()
        st.out = torch.empty_like(st.spec), torch.empty_like(st.real)
    elif kind == "mesh":
        st.pos, st.rho = _mesh_inputs(case, seed)
        st.out = torch.empty_like(st.rho), torch.empty((3, N, N, N), device="cuda")
    elif kind == "spectrum":
        st.out = [torch.empty((case["Np"] ** 3, 3), device="cuda") for _ in range(2)]
        _restore(st.sims[0], st.inp[0], n)
    else:
        st.out = [torch.empty((case["sims"], 3, case["Np"] ** 3), device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return st


def _restore(sim, state, n):
    s, v, acc = state
    pkg._check(pkg.lib().cola_import_state(sim.ctx, s.data_ptr(), v.data_ptr(), acc.data_ptr(), n, pkg.COLA_DEVICE), sim.ctx)


def run(st):
    case, kind, L = st.case, st.kind, pkg.lib()
    if kind == "job":
        with pkg.Simulation(st.run) as sim:
            sim.run_to_end()
            k, pk, nm = sim.pk()
            pkg._check(L.cola_export(sim.ctx, pkg.COLA_F_DISP, st.disp.data_ptr(), pkg.COLA_DEVICE), sim.ctx)
            sim.snapshot_device(None, st.vel)
        return {"k": k, "pk": pk.astype(np.float32), "modes": nm, "disp": st.disp, "vel": st.vel}  # P(k) is of a float32 mesh
    if kind == "transform":
        st.sims[0].fft_device(st.real, st.out[0], 1)
        st.sims[0].fft_device(st.spec, st.out[1], -1)
        return st.out
    if kind == "mesh":
        sim = st.sims[0]
        pkg._check(L.cola_cic_deposit(sim.ctx, st.pos.data_ptr(), st.pos.shape[0], st.out[0].data_ptr(), pkg.COLA_DEVICE), sim.ctx)
        sim.force_from_density_device(st.rho, 0.6, st.out[1])
        return st.out
    if kind == "spectrum":
        k, pk, nm = st.sims[0].pk(case["nbins"])
        st.sims[0].snapshot_device(*st.out)
        return {"k": k, "pk": pk.astype(np.float32), "modes": nm, "pos": st.out[0], "vel": st.out[1]}
    for sim, state in zip(st.sims, st.inp):
        _restore(sim, state, case["start"])
    if kind == "steps":
        st.sims[0].step(case["steps"])
    elif case["loop"]:
        for _ in range(case["steps"]):
            pkg.step_many(st.sims)
    else:
        with pkg.Batch(st.sims) as b:
            b.step(case["steps"])
    for which, out in zip((pkg.COLA_F_DISP, pkg.COLA_F_DV, pkg.COLA_F_ACC), st.out):
        for i, sim in enumerate(st.sims):
            pkg._check(L.cola_export(sim.ctx, which, out[i].data_ptr(), pkg.COLA_DEVICE), sim.ctx)
    return st.out


def work(case):
    """One HBM pass per array and per 3-D transform; five flops per point and level of a transform."""
    P, M, kind = float(case["Np"]) ** 3, float(case["Nmesh"]) ** 3, case["kind"]
    fft_p, fft_m = (2.5 * n * math.log2(n) for n in (P, M))
    if kind == "transform":
        return {"bytes": 16.0 * M, "flops": 2.0 * fft_m}
    if kind == "mesh":
        scr = bool(case["screening"])
        return {"bytes": 12.0 * case["npos"] + (4.0 + 16.0) * M, "flops": (6.0 if scr else 4.0) * fft_m + 30.0 * case["npos"]}
    if kind == "spectrum":
        return {"bytes": (12.0 + 12.0 + 24.0 + 8.0) * P + 8.0 * M, "flops": fft_m + 3.0 * fft_p + 60.0 * P}
    b = f = 0.0
    for _, _, _, scr in _models(case):
        steps = case["nsteps"] if kind == "job" else case["steps"]
        b += steps * (128.0 * P + (64.0 if scr else 40.0) * M) + 72.0 * P
        f += steps * ((6.0 if scr else 4.0) * fft_m + 6.0 * fft_p + 150.0 * P)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits

def _corners(x, N, L):
    """The eight CIC corners of positions x [3, P]: (flat cell index, weight)."""
    u = x * (N / L)
    i = u.floor()
    f = u - i
    i0 = [t.long() % N for t in i]
    for c in range(8):
        idx, w = 0, 1.0
        for d in (2, 1, 0):
            b = (c >> d) & 1
            idx = idx * N + (i0[d] + b) % N
            w = w * (f[d] if b else 1.0 - f[d])
        yield idx, w


def _deposit64(x, N, L):
    rho = torch.zeros(N**3, dtype=F64, device="cuda")
    for idx, w in _corners(x, N, L):
        rho.index_add_(0, idx, w)
    return rho.view(N, N, N)


def _force64(delta, L, a, model):
    """-grad Phi_tot of App. B with the screening of Sec. 6."""
    N = delta.shape[0]
    kind, fR0, rcH0, scr = model
    _, k2, g = _grid(N, L)
    dk = torch.fft.rfftn(delta)
    dk[0, 0, 0] = 0.0
    k2[0, 0, 0] = 1.0
    kap, C, am2 = 1.5 * OM * a, 0.0, 0.0
    if kind == FOFR:
        C, am2 = 1.0 / 3.0, a * a * _fr_m2(a, fR0)
    elif kind == NDGP:
        C = 1.0 / (3.0 * _dgp_beta(a, rcH0))
    if C and scr:
        if kind == FOFR:
            w = torch.fft.irfftn(dk * (-kap / (a * C_LIGHT) ** 2) / k2, s=(N, N, N)).abs_()
            eps = (1.5 * fR0 / _fr_x(a) ** 2 / w.clamp_min(1e-300)).clamp_max(1.0)
        else:
            w = torch.fft.irfftn(dk * torch.exp(-0.5 * k2), s=(N, N, N))
            x = 8.0 * rcH0**2 * OM / (9.0 * _dgp_beta(a, rcH0) ** 2) * (1.0 + w).clamp_min(0.0)
            eps = 2.0 / (torch.sqrt(1.0 + x) + 1.0)
        del w
        sk = torch.fft.rfftn(delta * eps)
        del eps
        sk[0, 0, 0] = 0.0
        dk += C * sk * (k2 / (k2 + am2))
        del sk
    elif C:
        dk *= 1.0 + C * (k2 / (k2 + am2))
    dk *= -kap / k2
    del k2
    return [torch.fft.irfftn(-1j * gi * dk, s=(N, N, N)) for gi in g]


def _lpt64(case, phi, c1, c2):
    """IFFT[i k (c1(k) phi1 + c2(k) phi2)] [3, P], the rows read by linear interpolation in ln k."""
    N, L = case["Np"], case["Lbox"]
    _, k2, g = _grid(N, L)
    lo, dl = _table_k(case)
    k2[0, 0, 0] = math.exp(2.0 * lo)
    u = (0.5 * k2.log() - lo) / dl
    i = u.floor().clamp(0, NK - 2).long()
    f = u - i
    sk = 0
    for row, p in zip((c1, c2), phi):
        t = torch.as_tensor(row, device="cuda")
        sk = sk + (t[i] * (1.0 - f) + t[i + 1] * f) * p
    return torch.stack([torch.fft.irfftn(1j * gi * sk, s=(N, N, N)).reshape(-1) for gi in g])


def _lattice64(case):
    N = case["Np"]
    q = torch.arange(N, dtype=F64, device="cuda") * (case["Lbox"] / N)
    return torch.stack([q.view(sh).expand(N, N, N).reshape(-1) for sh in ((1, 1, -1), (1, -1, 1), (-1, 1, 1))])


def _rows(case, model):
    lo, dl = _table_k(case)
    return _growth(model, _nodes(case), np.exp(lo + dl * np.arange(NK)))


def _steps64(case, model, rows, phi, state):
    """KDK steps of Sec. 2 in the frame of the LPT trajectory, from the float32 state."""
    s, v, acc = (x.double() for x in state)
    phi = [p.to(torch.complex128) for p in phi]
    a, N, L, q = _nodes(case), case["Nmesh"], case["Lbox"], _lattice64(case)
    for n in range(case["start"], case["start"] + case["steps"]):
        mid = 0.5 * (a[n] + a[n + 1])
        r0, r1 = rows[n], rows[n + 1]
        v = v + acc * _dtau(a[n], mid)
        s = s + v * _dtau(a[n], a[n + 1]) + _lpt64(case, phi, r1[0] - r0[0], r1[3] - r0[3])
        delta = _deposit64(q + s, N, L) * (N**3 / case["Np"] ** 3) - 1.0
        force = _force64(delta, L, a[n + 1], model)
        acc = -_lpt64(case, phi, r1[2], r1[5])
        for idx, w in _corners(q + s, N, L):
            for d in range(3):
                acc[d] += force[d].view(-1)[idx] * w
        v = v + acc * _dtau(mid, a[n + 1])
    return s, v, acc


def _spectrum64(x, N, L, Np, nbins):
    dk = torch.fft.rfftn(_deposit64(x, N, L) * (N**3 / Np**3) - 1.0)
    nf = torch.fft.fftfreq(N, 1.0 / N, dtype=F64, device="cuda")
    nh = torch.arange(N // 2 + 1, dtype=F64, device="cuda")
    win = [torch.sinc(t / N) ** 4 for t in (nf, nf, nh)]
    p = dk.abs() ** 2 * (L**3 / N**6) / (win[0].view(-1, 1, 1) * win[1].view(1, -1, 1) * win[2].view(1, 1, -1))
    n = torch.sqrt(nf.view(-1, 1, 1) ** 2 + nf.view(1, -1, 1) ** 2 + nh.view(1, 1, -1) ** 2)
    w = torch.full_like(nh, 2.0)
    w[0] = w[-1] = 1.0
    w = w.view(1, 1, -1).expand_as(n)
    b = torch.floor(n - 0.5).long()
    ok = (n >= 0.5) & (b < nbins)
    cnt, ps, ks = (torch.zeros(nbins, dtype=F64, device="cuda").index_add_(0, b[ok], t[ok]) for t in (w, w * p, w * n))
    return (ks / cnt * (2.0 * math.pi / L)).cpu().numpy(), (ps / cnt).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "job":
        return None  # its white noise is the library's own
    N, L = case["Nmesh"], case["Lbox"]
    if kind == "transform":
        gen = _generator(seed)
        real = torch.randn((N, N, N), generator=gen, device="cuda")
        spec = torch.fft.rfftn(torch.randn((N, N, N), generator=gen, device="cuda"))
        return torch.fft.rfftn(real.double()).contiguous(), torch.fft.irfftn(spec.to(torch.complex128), s=(N, N, N), norm="forward")
    if kind == "mesh":
        pos, rho = _mesh_inputs(case, seed)
        delta = rho.double() * (N**3 / case["Np"] ** 3) - 1.0
        return _deposit64(pos.double().T, N, L), torch.stack(_force64(delta, L, 0.6, _models(case)[0]))
    models = _models(case)
    rows = {m: _rows(case, m) for m in dict.fromkeys(models)}
    out = None
    for i, m in enumerate(models):
        phi = _potentials(case, _seed_of(seed, i))
        state = _state(case, _seed_of(seed, i), phi, case["start"])
        if kind == "spectrum":
            r = rows[m][case["start"]]
            x = _lattice64(case) + state[0].double()
            vel = (state[1].double() + _lpt64(case, phi, r[1], r[4])) * (100.0 / _nodes(case)[case["start"]])
            k, pk = _spectrum64(x, N, L, case["Np"], case["nbins"])
            x = x - L * torch.floor(x / L)
            return {"k": k, "pk": pk, "modes": None, "pos": x.T.contiguous(), "vel": vel.T.contiguous()}
        one = _steps64(case, m, rows[m], phi, state)
        if out is None:
            out = [torch.empty((case["sims"],) + tuple(t.shape), dtype=F64, device="cuda") for t in one]
        for o, t in zip(out, one):
            o[i] = t
    return out
