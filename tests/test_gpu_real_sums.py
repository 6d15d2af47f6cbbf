"""FP64 sums per ion in the real-space Ewald sum: partners whose forces cancel must not take the small terms summed
between them along.

Two unit charges at exactly one spacing on either side of an ion (coordinates and box powers of two: their separations
are exact and their forces cancel to the last bit), in columns of their own, and partners of charge 2^-17 in
others.  A pair term is FP32: each weak one is good to a few 1e-7 of itself, so the force on the middle ion is compared
at 1e-5 of the weak terms' magnitudes.  An FP32 sum that holds the unit term, 0.9, rounds at 3e-8 and leaves at least
1e-3 of the weak terms' 1e-6 to 1e-5.
"""
import numpy as np
import pytest

from oracle import ewald

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _box():
    rng = np.random.default_rng(11)
    middle = np.array([8.5, 8.5, 8.5])
    r = [middle, middle - [1.0, 0.0, 0.0], middle + [1.0, 0.0, 0.0]]
    for dx, dy in ((0, -2), (0, -1), (0, 1), (0, 2), (-2, 1), (-1, -2), (-1, 1), (1, -1), (1, 1), (2, 0)):
        r.append(middle + [dx, dy, 0.0] + rng.uniform(-0.4, 0.4, 3))
    q = np.full(len(r), 2.0 ** -17)
    q[:3] = 1.0
    return np.array(r), q


def test_weak_partners_between_cancelling_ones():
    from paper_2001_01583_gb300 import ewald_real_space_forces
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    L, rc, alpha = 16.0, 3.0, 0.5
    r, q = _box()
    want = ewald.real_space_forces(r, q, L, alpha, rc)[0]
    weak = [np.abs(ewald.real_space_forces(r[[0, j]], q[[0, j]], L, alpha, rc)[0]) for j in range(3, len(r))]
    F, _ = ewald_real_space_forces(torch.from_numpy(r), torch.from_numpy(q), L, alpha, rc)
    assert np.abs(F.cpu().numpy()[0] - want).max() <= 1e-5 * np.sum(weak, axis=0).max()
