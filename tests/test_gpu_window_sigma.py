"""The windows' polynomials where they converge slowest, cut-off 1 and the finest grids: 1-D plans at sigma = 4 and 16
against the formula in FP64.  Bars as in test_gpu_window_taps.py (1e-12 of the rms in FP64, 1e-5 in FP32): what the
polynomials leave out is at most 2.6e-16 and 4.1e-8 of the window's peak."""
import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WIN = {"gaussian": S.GAUSSIAN, "kaiser_bessel": S.KAISER_BESSEL, "sinc_power": S.SINC_POWER}


@pytest.mark.parametrize("window", list(WIN))
@pytest.mark.parametrize("sigma", [4.0, 16.0])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
def test_narrowest_windows_on_fine_grids(window, sigma, precision, tol):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N, M, m = (64,), 400, 1
    x = inputs.uniform_points(M, 1, seed=2)
    f, fh = inputs.complex_normal(M, seed=71), inputs.complex_normal(N, seed=72)
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    for sparse in (-1, 1 << 20):
        with Plan(N, M, sigma, m, window, precision) as p:
            p.set_option(_lib.OPT_SPARSE_POINTS, sparse)
            p.set_option(_lib.OPT_SPARSE_POINTS_INTERP, sparse)
            p.set_points(torch.from_numpy(x).cuda())
            a = p.adjoint(torch.from_numpy(f).to(dt).cuda())
            b = p.forward(torch.from_numpy(fh).to(dt).cuda())
            p.sync()
        for got, ref in ((a, S.adjoint(x, f, N, sigma, m, WIN[window])), (b, S.forward(x, fh, N, sigma, m, WIN[window]))):
            assert np.max(np.abs(got.cpu().numpy() - ref)) <= tol * np.sqrt(np.mean(np.abs(ref) ** 2))
