"""Small 1-D double-precision plans, whose transform is a direct sum over the chip, against the FP64 gridding oracle
(1e-12 of the rms per element, the bar of test_gpu_parity.py): lengths below a warp, ragged ones, and both sides of the
limit (N = 720 is the direct sum, N = 724 the FFT), one and several right-hand sides.
"""
import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [4, 6, 30, 64, 250, 720, 724])
@pytest.mark.parametrize("R,cap", [(1, 1), (3, 1), (5, 4)])
def test_direct_dft(N, R, cap):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    M, m = 333, 2 if N < 16 else 5
    x = inputs.uniform_points(M, 1, seed=N)
    f, fh = inputs.complex_normal((R, M), seed=91), inputs.complex_normal((R, N), seed=92)
    with Plan((N,), M, 2.0, m, "kaiser_bessel", "fp64") as p:
        if cap > 1:
            p.set_option(_lib.OPT_RHS_CAPACITY, cap)
        p.set_points(torch.from_numpy(x).cuda())
        a = p.adjoint(torch.from_numpy(f).cuda()).cpu().numpy()
        b = p.forward(torch.from_numpy(fh).cuda()).cpu().numpy()
        p.sync()
    for r in range(R):
        for got, ref in ((a[r], S.adjoint(x, f[r], (N,), 2.0, m, S.KAISER_BESSEL)),
                         (b[r], S.forward(x, fh[r], (N,), 2.0, m, S.KAISER_BESSEL))):
            assert np.max(np.abs(got - ref)) <= 1e-12 * np.sqrt(np.mean(np.abs(ref) ** 2))
