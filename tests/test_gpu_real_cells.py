"""Real-space Ewald sum with many ions and few partners (a thread per ion over cells): k^3 copies of a box side by side
have its forces and k^3 times its energy, against the oracle's direct sums over one box.  Cut-offs of few and of a few
hundred partners, boxes of more than 43 and of more than 128 cut-offs a side (the cells' number is then bounded), ions on
the box's faces and outside it, an ion without a position.

Bars as in test_gpu_real_columns.py: forces to 2e-5 of the largest, the energy to 1e-6 of the sum of the terms'
magnitudes.
"""
import numpy as np
import pytest

from oracle import ewald

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,rc,k,kind", [(700, 9.0, 2.5, 4, "random"),    # 63 partners, 44800 ions, 14 cut-offs a side
                                           (700, 9.0, 2.5, 5, "faces"),
                                           (400, 9.0, 0.8, 5, "random"),    # 1.2 partners, 56 cut-offs a side
                                           (40, 3.0, 0.35, 15, "random"),   # 129 cut-offs a side
                                           (1000, 6.0, 2.0, 4, "random")])  # 155 partners
def test_copies_of_a_box(n, L, rc, k, kind):
    from paper_2001_01583_gb300 import ewald_real_space, ewald_real_space_forces
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    alpha = 2.0 / rc
    rng = np.random.default_rng(n)
    r, q = rng.uniform(0.0, L, (n, 3)), rng.choice([-1.0, 2.0, 0.5], n)
    want = ewald.real_space_forces(r, q, L, alpha, rc)
    e, size = (ewald.real_space_energy(r, v, L, alpha, rc) for v in (q, np.abs(q)))
    shifts = L * np.stack(np.meshgrid(*[np.arange(float(k))] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    R, Q = (r + shifts).reshape(-1, 3), np.tile(q, k ** 3)
    if kind == "faces":   # whole boxes further out, and onto the faces from both sides
        R[::7] += k * L * rng.integers(-2, 3, (len(R[::7]), 3))
        R, Q = np.concatenate([R, [[np.nan, 1.0, 1.0]]]), np.concatenate([Q, [3.0]])
    F, got = ewald_real_space_forces(torch.from_numpy(R), torch.from_numpy(Q), k * L, alpha, rc)
    F = F.cpu().numpy()
    assert np.abs(F[:n * k ** 3].reshape(-1, n, 3) - want).max() <= 2e-5 * np.abs(want).max()
    assert np.all(F[n * k ** 3:] == 0.0)
    assert abs(got - k ** 3 * e) <= 1e-6 * k ** 3 * size
    assert abs(ewald_real_space(torch.from_numpy(R), torch.from_numpy(Q), k * L, alpha, rc) - k ** 3 * e) <= \
        1e-6 * k ** 3 * size
