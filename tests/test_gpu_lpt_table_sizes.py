"""Runs on 512^3 lattices whose growth tables differ in length take turns: the LPT z pass stages a single
run's table row in shared memory, so its launches differ in size."""
import numpy as np
import pytest

from workloads import LCDM_MODEL, Run

pytestmark = pytest.mark.gpu

BIG = Run(Np=512, Nmesh=64, Lbox=1024.0, nsteps=6, model=LCDM_MODEL)


def test_a_shorter_table_leaves_a_longer_one_usable():
    import paper_1703_00879_gb300 as pkg
    with pkg.Simulation(BIG.with_(nk_table=2048)) as a, pkg.Simulation(BIG.with_(nk_table=16, seed=1)) as b:
        a.step(1)
        b.step(1)
        a.step(1)
        assert a.steps_done == 2 and a.check_state() == 0


def test_a_table_that_does_not_fit_in_shared_memory():
    """A single run reads such a row from global memory, as grouped runs read every row: the same
    fields bit for bit."""
    import paper_1703_00879_gb300 as pkg
    runs = [BIG.with_(nk_table=8192, seed=s) for s in (0, 1)]
    with pkg.Simulation(runs[0]) as solo:
        solo.step(1)
        fields = [solo.export(w) for w in (pkg.COLA_F_LPT_DISP, pkg.COLA_F_LPT_ACC)]
    sims = [pkg.Simulation(r, ic=False) for r in runs]
    pkg.ic_many(sims)
    pkg.step_many(sims)
    for f, w in zip(fields, (pkg.COLA_F_LPT_DISP, pkg.COLA_F_LPT_ACC)):
        assert np.array_equal(f, sims[0].export(w))
    for s in sims:
        s.close()
