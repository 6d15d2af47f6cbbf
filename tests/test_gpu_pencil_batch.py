"""Batch items of many grid sizes share the pencil launches: every item element by element against the FP64 gridding
oracle (1e-5 of the rms, test_gpu_batch.py's bar), grids smaller than a pencil's tile and items left to the other kernels
among them, and no more launches than the same batch of equal sizes."""
import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _launches(Ns, Ms):
    from paper_2001_01583_gb300 import Batch
    xs = [inputs.uniform_points(M, 3, seed=i) for i, M in enumerate(Ms)]
    fs = [inputs.complex_normal((1, M), seed=50 + i) for i, M in enumerate(Ms)]
    hs = [inputs.complex_normal((1,) + N, seed=70 + i) for i, N in enumerate(Ns)]
    with Batch([dict(N=N, M=M) for N, M in zip(Ns, Ms)], "fp32") as b:
        b.set_points([torch.from_numpy(x).cuda() for x in xs])
        before = b.kernel_launches()
        A = b.adjoint([torch.from_numpy(f).to(torch.complex64).cuda() for f in fs])
        B = b.forward([torch.from_numpy(h).to(torch.complex64).cuda() for h in hs])
        b.sync()
        launches = b.kernel_launches() - before
    for i, N in enumerate(Ns):
        for got, ref in ((A[i][0], S.adjoint(xs[i], fs[i][0], N, 2.0, 4, S.KAISER_BESSEL)),
                         (B[i][0], S.forward(xs[i], hs[i][0], N, 2.0, 4, S.KAISER_BESSEL))):
            d = np.abs(got.cpu().numpy() - ref)
            assert np.max(d) <= 1e-5 * np.sqrt(np.mean(np.abs(ref) ** 2)), i
    return launches


def test_items_of_many_sizes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Ns = [(6, 6, 6), (8, 20, 12), (24, 10, 16), (16, 16, 16), (30, 6, 8), (12, 12, 40)]
    Ms = [40, 900, 1500, 2000, 300, 2500]
    assert _launches(Ns, Ms) == 4
    _launches([(16, 16, 16), (32, 32, 32)], [3000, 200])   # the second below a point per plane
