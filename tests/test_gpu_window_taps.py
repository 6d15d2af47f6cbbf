"""The windows' polynomials (window_taps, window_tap) against the formula in FP64: 1-D plans, narrow to wide windows,
with points on grid nodes (offset 0, where a cut window's last tap is 0) and just below the next node.

Bars as in test_gpu_parity.py: element by element against the FP64 gridding oracle, 1e-12 of the rms in FP64 and 1e-5
in FP32 (windows whose scaling factor stays small: m <= 8).
"""
import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WIN = {"gaussian": S.GAUSSIAN, "kaiser_bessel": S.KAISER_BESSEL, "sinc_power": S.SINC_POWER}


@pytest.mark.parametrize("window,m,precision", [(w, m, p) for w in WIN for m, p in
                                                [(1, "fp64"), (2, "fp64"), (5, "fp64"), (12, "fp64"),
                                                 (1, "fp32"), (2, "fp32"), (8, "fp32")]])
@pytest.mark.parametrize("sparse", [-1, 1 << 20])
def test_polynomial_windows(window, m, precision, sparse):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N, M = (64,), 400
    x = inputs.uniform_points(M, 1, seed=m)
    x[:40, 0] = np.arange(-20, 20) / 128.0              # nodes of the 128-cell grid, exact in binary
    x[40:60, 0] = (np.arange(20) + 1 - 2.0 ** -12) / 128.0
    f, fh = inputs.complex_normal(M, seed=71), inputs.complex_normal(N, seed=72)
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    with Plan(N, M, 2.0, m, window, precision) as p:
        p.set_option(_lib.OPT_SPARSE_POINTS, sparse)         # a tile, or a warp per point on the grid
        p.set_option(_lib.OPT_SPARSE_POINTS_INTERP, sparse)
        p.set_points(torch.from_numpy(x).cuda())
        a = p.adjoint(torch.from_numpy(f).to(dt).cuda())
        b = p.forward(torch.from_numpy(fh).to(dt).cuda())
        p.sync()
    tol = 1e-12 if precision == "fp64" else 1e-5
    for got, ref in ((a, S.adjoint(x, f, N, 2.0, m, WIN[window])), (b, S.forward(x, fh, N, 2.0, m, WIN[window]))):
        err = np.max(np.abs(got.cpu().numpy() - ref)) / np.sqrt(np.mean(np.abs(ref) ** 2))
        assert err <= tol, (window, m, err)


@pytest.mark.parametrize("window", list(WIN))
def test_offsets_within_rounding_of_a_node(window):
    """A narrow FP32 window is cut where the formula's rounded argument reaches the cut: the kernels that take the
    polynomials (a tile) against the one that takes the formula (a warp per point), 1e-5 of the rms; a tap that one of
    them keeps would be 1e-3."""
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N, M = (64,), 60
    x = ((np.arange(M) - 30) / 128.0 + np.repeat([2.0 ** -34, -2.0 ** -34, 2.0 ** -40], 20))[:, None]
    f, fh = inputs.complex_normal(M, seed=73), inputs.complex_normal(N, seed=74)
    out = []
    for sparse in (-1, 1 << 20):
        with Plan(N, M, 2.0, 2, window, "fp32") as p:
            p.set_option(_lib.OPT_SPARSE_POINTS, sparse)
            p.set_option(_lib.OPT_SPARSE_POINTS_INTERP, sparse)
            p.set_points(torch.from_numpy(x).cuda())
            a = p.adjoint(torch.from_numpy(f).to(torch.complex64).cuda())
            b = p.forward(torch.from_numpy(fh).to(torch.complex64).cuda())
            p.sync()
            out.append((a.cpu().numpy(), b.cpu().numpy()))
    for got, ref in zip(*out):
        assert np.max(np.abs(got - ref)) <= 1e-5 * np.sqrt(np.mean(np.abs(ref) ** 2)), window
