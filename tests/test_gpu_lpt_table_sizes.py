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
