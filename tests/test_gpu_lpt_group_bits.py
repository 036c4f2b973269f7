"""A lattice's LPT fields do not depend on how many lattices share the launch: the initial conditions of
cola_ic_many and the fields of a grouped step equal those of the context alone, bit for bit (no
atomics on that path), also where the group is large enough for the register-resident LPT z pass
while the lattice alone takes the short-chain one."""
import numpy as np
import pytest

from workloads import ensemble_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Np,n", [(32, 40), (64, 16), (128, 4)])
def test_fields_alone_and_in_a_large_group(Np, n):
    import paper_1703_00879_gb300 as pkg
    runs = [ensemble_run(seed, Np=Np, Nmesh=Np, Lbox=2.0 * Np, nsteps=4) for seed in range(n)]
    sims = [pkg.Simulation(r, ic=False) for r in runs]
    pkg.ic_many(sims)
    some = (0, 1, 2, n - 1)
    first = [sims[i].export(pkg.COLA_F_DISP) for i in some]
    pkg.step_many(sims)
    for i, d in zip(some, first):
        with pkg.Simulation(runs[i]) as solo:
            assert np.array_equal(d, solo.export(pkg.COLA_F_DISP))
            if i == 0:  # the group's first context exports the fields of the grouped step
                solo.step(1)
                for which in (pkg.COLA_F_LPT_DISP, pkg.COLA_F_LPT_ACC):
                    assert np.array_equal(sims[0].export(which), solo.export(which))
    for s in sims:
        s.close()
