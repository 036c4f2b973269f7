"""The two forms of the LPT z pass give the same fields: a lattice of 32^3 or 64^3 alone takes the
short-chain kernel, the same lattice in a large cola_ic_many group the register-resident one.

Tolerance: both form the same products with at most two differently fused roundings per mode and
transform level (u = 6e-8), an independent error of 2 u sqrt(2 log2(N^3)) < 8e-7 of the field's rms,
below 5e-6 of its largest value at any of N^3 points."""
import numpy as np
import pytest

from workloads import ensemble_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Np,n", [(32, 40), (64, 16)])
def test_lpt_fields_alone_and_in_a_group(Np, n):
    import paper_1703_00879_gb300 as pkg
    runs = [ensemble_run(seed, Np=Np, Nmesh=Np, Lbox=2.0 * Np, nsteps=4) for seed in range(n)]
    sims = [pkg.Simulation(r, ic=False) for r in runs]
    pkg.ic_many(sims)
    for i in (0, 1, 2, n - 1):
        with pkg.Simulation(runs[i]) as solo:
            a, b = sims[i].export(pkg.COLA_F_DISP), solo.export(pkg.COLA_F_DISP)  # the fields at a_ini
            assert np.max(np.abs(a - b)) <= 5e-6 * np.max(np.abs(b))
    for s in sims:
        s.close()
