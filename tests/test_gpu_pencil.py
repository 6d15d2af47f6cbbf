"""The 3-D single-precision pencil kernels (automatic method, a point per pencil plane or more) element by element
against the FP64 gridding oracle: every window width, ragged grids smaller and larger than a pencil's tile, points
spread out and packed into few cells (the dense form), several right-hand sides, subproblem sizes that cut planes.

Bars as for the wide windows in test_gpu_parity.py: rounding on the grid reaches the adjoint's outputs multiplied by the
scaling factor c_0 / c_k, so they are compared with that factor taken out at 1e-5 of the rms (FP32 weights and sums), and
the forward's, whose input is multiplied by it, at 1e-5 times the factor's rms.
"""
import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WIN = {"gaussian": S.GAUSSIAN, "kaiser_bessel": S.KAISER_BESSEL, "sinc_power": S.SINC_POWER}


def _check(N, x, m, window, sub, R=1):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    M = x.shape[0]
    f, fh = inputs.complex_normal((R, M), seed=81), inputs.complex_normal((R,) + N, seed=82)
    with Plan(N, M, 2.0, m, window, "fp32") as p:
        if sub:
            p.set_option(_lib.OPT_MAX_SUBPROBLEM, sub)
        if R > 1:
            p.set_option(_lib.OPT_RHS_CAPACITY, R)
        p.set_points(torch.from_numpy(x).cuda())
        a = p.adjoint(torch.from_numpy(f).to(torch.complex64).cuda())
        b = p.forward(torch.from_numpy(fh).to(torch.complex64).cuda())
        p.sync()
        n = p.info()["n"]
    amp = np.ones(())
    for w in S.scaling_weights(WIN[window], m, list(N), list(n)):
        amp = np.multiply.outer(amp, np.abs(w).max() / np.abs(w))
    for r in range(R):
        for got, ref, by, bar in ((a[r], S.adjoint(x, f[r], N, 2.0, m, WIN[window]), amp, 1e-5),
                                  (b[r], S.forward(x, fh[r], N, 2.0, m, WIN[window]), 1.0,
                                   1e-5 * np.sqrt(np.mean(amp ** 2)))):
            d = np.abs(got.cpu().numpy() - ref) / by
            assert np.max(d) <= bar * np.sqrt(np.mean(np.abs(ref) ** 2))


@pytest.mark.parametrize("window,m", [("kaiser_bessel", m) for m in range(1, 9)] + [("gaussian", 3), ("gaussian", 7),
                                                                                  ("sinc_power", 4)])
@pytest.mark.parametrize("kind,sub", [("uniform", 0), ("uniform", 200), ("packed", 1024), ("packed", 2000)])
def test_pencils(window, m, kind, sub):
    N = (20, 12, 26)
    x = inputs.uniform_points(3000, 3, seed=m) if kind == "uniform" else inputs.clustered_points(3000, 3, 3, 0.004, m)
    _check(N, x, m, window, sub)


@pytest.mark.parametrize("N,M,m,R", [((6, 6, 6), 1, 1, 1), ((6, 8, 10), 700, 2, 1), ((600, 8, 8), 4000, 4, 1),
                                     ((10, 34, 18), 5000, 4, 3), ((16, 12, 14), 9000, 6, 2)])
def test_pencil_shapes(N, M, m, R):
    x = inputs.uniform_points(M, 3, seed=5)
    x[0] = -0.5                          # the corner: every dimension wraps
    _check(N, x, m, "kaiser_bessel", 0, R)
