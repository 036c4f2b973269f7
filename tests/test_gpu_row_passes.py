"""The x passes (real rows to half spectra and back) at every length the library takes, inside the
3-D transforms of cola_fft on device arrays, against double-precision FFTs.

Tolerance: each of the L = log2(N^3) radix-2 levels and the real split rounds once or twice with
unit roundoff u = 6e-8; independent roundings add to at most 2 u sqrt(L + 2) of the 2-norm
(L <= 30: 7e-7)."""
import pytest
import torch

from workloads import SMALL_F5

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32, 64, 128, 256, 512, 1024])
def test_real_transforms_against_double_precision(N):
    import paper_1703_00879_gb300 as pkg
    run = SMALL_F5.with_(Nmesh=N, Lbox=float(N))
    gen = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn((N, N, N), generator=gen, device="cuda")
    X = torch.empty((N, N, N // 2 + 1), dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    with pkg.Simulation(run, ic=False) as sim:
        sim.fft_device(x, X, 1)
        sim.fft_device(X, y, -1)
        ref = torch.fft.rfftn(x.double())
        for part in (slice(None), (slice(None), slice(None), 0), (slice(None), slice(None), N // 2)):
            a, b = X[part].to(torch.complex128), ref[part]
            assert torch.linalg.vector_norm(a - b) <= 7e-7 * torch.linalg.vector_norm(b)
        back = torch.fft.irfftn(X.to(torch.complex128), s=(N, N, N), norm="forward")
        assert torch.linalg.vector_norm(y.double() - back) <= 7e-7 * torch.linalg.vector_norm(back)
