"""The y derivative of the LPT fields rounds its products i ky X(ky) once each, before the y inverse
transform, at every lattice length and in whichever pass it runs.

The 16-bit per-step fields take their scales from these fields: a product that is fused with the
transform's first additions moves a scale by one unit in the last place and with it up to one code of
every value (2^-8 of it with bf16).

How the rounding is seen: potentials with modes at kz = +1 only are their own z inverse on the plane
z = 0, with no rounding.  For A with modes at ky = 0, +-1, +-2, +-4, ... and B = ky A the field
Psi_y of A is there the y inverse of the rounded products i (kf ky) X, and Psi_z of B that of the
rounded products i kf (ky X): the same values, since ky is a power of two and |k| (the growth
coefficients) is the same.  So the two fields are equal bit for bit."""
import numpy as np
import pytest

from workloads import LCDM_MODEL, Run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32, 64, 128, 256, 512])
def test_y_derivative_products_are_rounded_once(N):
    import paper_1703_00879_gb300 as pkg
    run = Run(Np=N, Nmesh=N, Lbox=1.7 * N, nsteps=4, model=LCDM_MODEL)
    rng = np.random.default_rng(N)
    ky = np.array([0] + [s * 2**j for j in range(N.bit_length() - 2) for s in (1, -1)])
    x = rng.standard_normal((ky.size, N // 2 + 1, 2)).astype(np.float32) * np.float32(run.Lbox / N)
    x = x[..., 0] + 1j * x[..., 1]
    fields = []
    for values, which in ((x, 1), (x * ky[:, None].astype(np.float32), 2)):
        phi = np.zeros((N, N, N // 2 + 1), np.complex64)
        phi[1, ky] = values
        with pkg.Simulation(run, phi=(phi, np.zeros_like(phi))) as s:
            psi = s.export(pkg.COLA_F_LPT_DISP)
        fields.append(psi.reshape(3, N, N, N)[which, 0])
    assert np.max(np.abs(fields[0])) > 0
    assert np.array_equal(fields[0], fields[1])
