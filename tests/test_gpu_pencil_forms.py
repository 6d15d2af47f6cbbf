"""Interpolation of pencils with few points per plane: from the grid point by point, from slabs, or both, by the points'
density.  Element by element against the FP64 gridding oracle, every window width, uniform points around the density at
which the form changes, clusters in a sparse background, several right-hand sides, pencils cut along dimension 0
(n_0 > 1023), and the two forms against one another in a batch.

Bars as in test_gpu_pencil.py: rounding on the grid reaches the adjoint's outputs multiplied by the scaling factor
c_0 / c_k, so they are compared with that factor taken out at 1e-5 of the rms, and the forward's at 1e-5 times the
factor's rms.
"""
import math

import numpy as np
import pytest

from oracle import nfft_steps as S
from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGE = {1: 15, 2: 13, 3: 11, 4: 9, 5: 7, 6: 13, 7: 11, 8: 9}   # cells of a pencil's cross-section per side


def _bars(N, n, m):
    amp = np.ones(())
    for w in S.scaling_weights(S.KAISER_BESSEL, m, list(N), list(n)):
        amp = np.multiply.outer(amp, np.abs(w).max() / np.abs(w))
    return amp


def _check(N, x, m, R=1):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    M = x.shape[0]
    f, fh = inputs.complex_normal((R, M), seed=81), inputs.complex_normal((R,) + N, seed=82)
    with Plan(N, M, 2.0, m, "kaiser_bessel", "fp32") as p:
        if R > 1:
            p.set_option(_lib.OPT_RHS_CAPACITY, R)
        p.set_points(torch.from_numpy(x).cuda())
        a = p.adjoint(torch.from_numpy(f).to(torch.complex64).cuda())
        b = p.forward(torch.from_numpy(fh).to(torch.complex64).cuda())
        p.sync()
        info = p.info()
    assert info["bin"][0] == 1023            # pencils
    amp = _bars(N, info["n"], m)
    for r in range(R):
        for got, ref, by, bar in ((a[r], S.adjoint(x, f[r], N, 2.0, m, S.KAISER_BESSEL), amp, 1e-5),
                                  (b[r], S.forward(x, fh[r], N, 2.0, m, S.KAISER_BESSEL), 1.0,
                                   1e-5 * np.sqrt(np.mean(amp ** 2)))):
            d = np.abs(got.cpu().numpy() - ref) / by
            assert np.max(d) <= bar * np.sqrt(np.mean(np.abs(ref) ** 2))


def _points(n, m, density):
    return math.ceil(density * n[0] * n[1] * n[2] / EDGE[m] ** 2)


@pytest.mark.parametrize("m", range(1, 9))
@pytest.mark.parametrize("density,R", [(1.02, 1), (2.2, 2), (4.5, 1)])
def test_uniform_densities(m, density, R):
    N = (24, 18, 20)
    _check(N, inputs.uniform_points(_points([2 * v for v in N], m, density), 3, seed=m), m, R)


@pytest.mark.parametrize("m", range(1, 9))
@pytest.mark.parametrize("share", [0.3, 0.8])
def test_clusters_in_a_background(m, share):
    """Dense and sparse subproblems of one set, either holding most of the points."""
    N = (24, 18, 20)
    M = _points([2 * v for v in N], m, 1.2)
    k = int(share * M)
    x = np.concatenate([inputs.clustered_points(k, 3, 3, 0.004, m), inputs.uniform_points(M - k, 3, seed=m)])
    _check(N, x[np.random.default_rng(m).permutation(M)], m)


@pytest.mark.parametrize("m,N,density,R", [(1, (524, 6, 8), 1.1, 1), (3, (524, 6, 8), 1.3, 2), (3, (524, 6, 8), 3.0, 1),
                                           (6, (524, 8, 8), 1.1, 3), (6, (524, 8, 8), 6.0, 1), (8, (524, 10, 10), 1.5, 1)])
def test_pencils_cut_along_dimension_0(m, N, density, R):
    x = inputs.uniform_points(_points([1050] + [2 * v for v in N[1:]], m, density), 3, seed=5)
    x[:40, 0] = (np.arange(40) - 20 + 1023.4) / 1050.0   # around the cut at plane 1023 of 1050
    _check(N, x - np.floor(x + 0.5), m, R)


def test_batch_items_of_either_form():
    """Items below and above the density share their launches: each has the results it has as a plan of its own."""
    from paper_2001_01583_gb300 import Batch, Plan
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    m, Ns = 6, [(20, 20, 20), (24, 18, 22), (16, 16, 16)]
    Ms = [_points([2 * v for v in N], m, d) for N, d in zip(Ns, (1.1, 3.0, 2.0))]
    xs = [torch.from_numpy(inputs.uniform_points(M, 3, seed=i)).cuda() for i, M in enumerate(Ms)]
    xs[2] = torch.from_numpy(inputs.clustered_points(Ms[2], 3, 2, 0.004, 3)).cuda()
    hs = [torch.from_numpy(inputs.complex_normal((1,) + N, seed=70 + i)).to(torch.complex64).cuda()
          for i, N in enumerate(Ns)]
    with Batch([dict(N=N, M=M) for N, M in zip(Ns, Ms)], "fp32", m=m) as b:
        b.set_points(xs)
        out = b.forward(hs)
        b.sync()
    for N, M, x, h, got in zip(Ns, Ms, xs, hs, out):
        with Plan(N, M, 2.0, m, "kaiser_bessel", "fp32") as p:
            p.set_points(x)
            want = p.forward(h)
            p.sync()
        amp = _bars(N, [2 * v for v in N], m)
        rms = float(want.abs().square().mean().sqrt())
        assert float((got - want).abs().max()) <= 2e-5 * np.sqrt(np.mean(amp ** 2)) * rms
