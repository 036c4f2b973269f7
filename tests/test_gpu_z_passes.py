"""The fused force-side z passes (forward transform, k-space operation and inverse transforms on one
tile) above the mesh sizes of test_gpu_parity.py: the mesh force of a given density against the FP64
oracle, each model family and screening state, on meshes of 256 and 512 points.

Tolerance: the force passes round each value about 2 log2(N^3) + 20 times (two to four transforms
and the per-mode factors) with unit roundoff 6e-8 relative to the field's rms; the largest error over
N^3 cells is about six standard deviations of that random walk, 6 x 6e-8 sqrt(74) = 3.1e-6 of the
rms, below 1e-5 of the largest force."""
import numpy as np
import pytest

from oracle import pm
from workloads import F5, F5_NOSCREEN, LCDM_MODEL, NDGP1, Run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,model", [(256, LCDM_MODEL), (256, F5), (256, NDGP1), (512, F5), (512, F5_NOSCREEN)],
                         ids=["256_lcdm", "256_F5", "256_nDGP", "512_F5", "512_F5_unscreened"])
def test_force_of_a_density(N, model):
    import paper_1703_00879_gb300 as pkg
    run = Run(Np=32, Nmesh=N, Lbox=16.0 * N, nsteps=4, model=model)
    rng = np.random.default_rng(N)
    mean = 32.0**3 / N**3
    rho = (mean * np.exp(rng.standard_normal((N, N, N), dtype=np.float32) - 0.5)).astype(np.float32)
    a = 0.6
    with pkg.Simulation(run, ic=False) as s:
        F = s.force_from_density(rho, a)
    ref = pm.force_mesh(rho.astype(np.float64), mean, N, run.Lbox, a, run.cosmo.Omega_m, model)
    for i in range(3):
        assert np.max(np.abs(F[i] - ref[i])) <= 1e-5 * np.max(np.abs(ref[i])), i
