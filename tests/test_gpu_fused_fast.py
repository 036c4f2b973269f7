"""Multi-step calls on the scale-independent LPT path join the kick of each step with the drift and
deposit of the next, both from one read of Psi1 and Psi2 (Sec. 4.1 with D(k, a) = D(a)): K steps in
one call equal K calls of one step.

Tolerance: the two differ in the order of the deposit's float additions and in which products of the
two-term combinations are fused (a few units of 6e-8 of each field per step); over ten steps below
1e-5 of the largest value, and 1e-4 cell as for the fused per-k path."""
import numpy as np
import pytest

from workloads import LCDM_MODEL, NDGP1, SMALL_F5

pytestmark = pytest.mark.gpu


def _run(pkg, run, calls, **kw):
    with pkg.Simulation(run, lpt_fast=True, **kw) as s:
        for k in calls:
            s.step(k)
        return [s.export(w).astype(np.float64) for w in (pkg.COLA_F_DISP, pkg.COLA_F_DV, pkg.COLA_F_ACC,
                                                         pkg.COLA_F_LPT_DISP, pkg.COLA_F_LPT_ACC)]


@pytest.mark.parametrize("model,Nmesh,prec", [(LCDM_MODEL, 32, 0), (NDGP1, 64, 0), (LCDM_MODEL, 32, 2)],
                         ids=["lcdm", "ndgp", "lcdm_fp16_seeds"])
def test_fused_fast_steps_equal_single_steps(model, Nmesh, prec):
    import paper_1703_00879_gb300 as pkg
    run = SMALL_F5.with_(model=model, Nmesh=Nmesh)
    ref = _run(pkg, run, [1] * 10, seed_precision=prec)
    for calls in ([10], [2, 1, 7]):
        got = _run(pkg, run, calls, seed_precision=prec)
        cell = run.Lbox / run.Nmesh
        assert np.max(np.abs(got[0] - ref[0])) <= 1e-4 * cell
        for a, b in zip(got[1:], ref[1:]):
            assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b))


def test_fused_fast_boundary_on_the_paired_force_mesh():
    """The same boundary with the interleaved force pairs (meshes above 128 points).  Two steps only: on
    a mesh eight times finer than the lattice two runs of the same calls differ by 1e-3 cell after
    ten steps (the order of the deposit's additions, amplified by close encounters), and by at most
    4e-6 cell after two or three."""
    import paper_1703_00879_gb300 as pkg
    run = SMALL_F5.with_(model=LCDM_MODEL, Nmesh=256)
    ref, got = _run(pkg, run, [1, 1]), _run(pkg, run, [2])
    assert np.max(np.abs(got[0] - ref[0])) <= 1e-4 * run.Lbox / run.Nmesh
    for a, b in zip(got[1:], ref[1:]):
        assert np.max(np.abs(a - b)) <= 1e-4 * np.max(np.abs(b))
