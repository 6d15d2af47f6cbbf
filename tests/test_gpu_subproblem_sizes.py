"""The automatic subproblem size: a bin's pieces are as even as can be.  The results are those of an explicit size (the
order of the atomic sums apart: 1e-5 of the rms in FP32, 1e-12 in FP64) and of the FP64 gridding oracle
(test_gpu_parity.py's bars), over the kernels of 1 to 3 dimensions, for uniform and clustered points, bins of one point
more than a piece, and more bins than the one-block kernel takes.
"""
import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("N,M,kind", [((256, 250), 40000, "uniform"), ((256, 250), 40000, "clustered"),
                                      ((256, 256), 40000, "edge"), ((2100, 2100), 30000, "clustered"),
                                      ((4096,), 30000, "uniform"),
                                      ((4096,), 30000, "clustered"), ((40, 40, 40), 20000, "uniform"),
                                      ((40, 40, 40), 20000, "clustered")])
def test_automatic_size(N, M, kind, precision, tol):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d, m = len(N), 4
    x = inputs.uniform_points(M, d, seed=1) if kind != "clustered" else inputs.clustered_points(M, d, 4, 0.01, 1)
    if kind == "edge":   # bins of 101 and of 1025 points and no others: a piece and a point
        x = 0.05 * x - 0.47
        x[:1025] += 0.25
        x[1025:1126] += 0.125
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    f, fh = inputs.complex_normal(M, seed=71), inputs.complex_normal(N, seed=72)
    out = []
    for size in (0, 1024, 100):
        with Plan(N, M, 2.0, m, "kaiser_bessel", precision) as p:
            if size:
                p.set_option(_lib.OPT_MAX_SUBPROBLEM, size)
            if d == 3:
                p.set_option(_lib.OPT_BIN_0, 8)   # not pencils
            p.set_points(torch.from_numpy(x).cuda())
            out.append((p.adjoint(torch.from_numpy(f).to(dt).cuda()).cpu().numpy(),
                        p.forward(torch.from_numpy(fh).to(dt).cuda()).cpu().numpy()))
            p.sync()
    refs = (S.adjoint(x, f, N, 2.0, m, S.KAISER_BESSEL), S.forward(x, fh, N, 2.0, m, S.KAISER_BESSEL))
    for k, ref in enumerate(refs):
        rms = np.sqrt(np.mean(np.abs(ref) ** 2))
        assert np.max(np.abs(out[0][k] - ref)) <= tol * rms
        for other in out[1:]:
            assert np.max(np.abs(out[0][k] - other[k])) <= tol * rms
