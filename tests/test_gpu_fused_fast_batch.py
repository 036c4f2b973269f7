"""The joined step boundaries of the scale-independent LPT path: that multi-step calls take them, and
that a Batch of several runs takes them with the results of single steps.

Tolerance: as for the single runs (the order of the deposit's float additions and the fusing of
the two-term products, a few units of 6e-8 per step): 1e-4 cell, 1e-4 of the largest value."""
import numpy as np
import pytest

from workloads import LCDM_MODEL, NDGP1, SMALL_F5

pytestmark = pytest.mark.gpu

RUN = SMALL_F5.with_(nsteps=6)


def _boundaries(pkg, call):
    """Launches of the joined boundary pass and of the separate kick in call(sim)."""
    with pkg.Simulation(RUN.with_(model=LCDM_MODEL), lpt_fast=True) as s:
        s.profile()
        call(s)
        stages = s.profile_read()
    return stages["kick_drift_deposit"][1], stages["gather_kick"][1]


def test_multi_step_calls_join_the_boundaries():
    import paper_1703_00879_gb300 as pkg
    assert _boundaries(pkg, lambda s: s.step(6)) == (5, 1)
    assert _boundaries(pkg, lambda s: [s.step(1) for _ in range(6)]) == (0, 6)

    def batch(s):
        with pkg.Batch([s]) as b:
            b.step(6)

    assert _boundaries(pkg, batch) == (5, 1)


@pytest.mark.parametrize("Nmesh", [32, 256], ids=["components", "pairs"])
def test_batch_steps_equal_single_steps(Nmesh):
    import paper_1703_00879_gb300 as pkg
    runs = [RUN.with_(model=m, seed=i, Nmesh=Nmesh) for i, m in enumerate((LCDM_MODEL, NDGP1, LCDM_MODEL))]
    which = (pkg.COLA_F_DISP, pkg.COLA_F_DV, pkg.COLA_F_ACC)
    steps = 2 if Nmesh > 128 else 6  # a mesh this much finer than the lattice is chaotic over more
    want = []
    for r in runs:
        with pkg.Simulation(r, lpt_fast=True) as s:
            for _ in range(steps):
                s.step(1)
            want.append([s.export(w).astype(np.float64) for w in which])
    sims = [pkg.Simulation(r, lpt_fast=True) for r in runs]
    with pkg.Batch(sims) as b:
        b.step(steps)
    for r, s, ref in zip(runs, sims, want):
        got = [s.export(w).astype(np.float64) for w in which]
        assert np.max(np.abs(got[0] - ref[0])) <= 1e-4 * r.Lbox / r.Nmesh
        for a, c in zip(got[1:], ref[1:]):
            assert np.max(np.abs(a - c)) <= 1e-4 * np.max(np.abs(c))
        s.close()
