"""The column form of the real-space Ewald sum (boxes of three cut-offs and more) against the oracle's direct sums:
single ions and pairs, counts around a warp's ions, boxes of exactly and just over three cut-offs, empty columns, ions on
the box's faces and outside it, columns filled unevenly along z.

Bars as in test_gpu_forces.py and test_gpu_ewald.py: forces to 2e-5 of the largest, the energy to 1e-6 of the sum of the
terms' magnitudes (FP32 pair terms and sums).
"""
import numpy as np
import pytest

from oracle import ewald

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ions(n, L, kind, seed):
    rng = np.random.default_rng(seed)
    r = rng.uniform(0.0, L, (n, 3))
    if kind == "faces":
        r[::3, 0] = 0.0
        r[1::3, 2] = np.nextafter(L, 0.0)
        r[2::5] += L * rng.integers(-2, 3, (len(r[2::5]), 3))
    elif kind == "columns":                       # few columns, ions bunched at both ends of z
        r[:, :2] = L * (np.floor(rng.uniform(0, 3, (n, 2))) + 0.3) / 3 + 0.2 * rng.random((n, 2))
        r[:, 2] = np.where(rng.random(n) < 0.5, 0.3 * rng.random(n), L - 0.4 * rng.random(n))
    return r, rng.choice([-1.0, 2.0, 0.5], n)


@pytest.mark.parametrize("n,L,rc,kind", [(1, 9.0, 3.0, "random"), (2, 9.0, 3.0, "random"), (9, 9.1, 3.0, "faces"),
                                         (65, 10.0, 3.3, "columns"), (400, 9.0, 3.0, "faces"),
                                         (700, 30.0, 2.0, "random"), (300, 12.0, 2.5, "columns")])
def test_columns(n, L, rc, kind):
    from paper_2001_01583_gb300 import ewald_real_space, ewald_real_space_forces
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    alpha = 0.8
    r, q = _ions(n, L, kind, n)
    want = ewald.real_space_forces(r, q, L, alpha, rc)
    size = ewald.real_space_energy(r, np.abs(q), L, alpha, rc)
    e = ewald.real_space_energy(r, q, L, alpha, rc)
    F, got = ewald_real_space_forces(torch.from_numpy(r), torch.from_numpy(q), L, alpha, rc)
    assert np.abs(F.cpu().numpy() - want).max() <= 2e-5 * max(np.abs(want).max(), 1e-300)
    assert abs(got - e) <= 1e-6 * size
    assert abs(ewald_real_space(torch.from_numpy(r), torch.from_numpy(q), L, alpha, rc) - e) <= 1e-6 * size


@pytest.mark.parametrize("n", [720, 721, 1081, 1443])
def test_ions_per_warp(n):
    """2, 4, 6 and 8 ions per warp: 27 copies of a box (a cube of 3 on a side) have its forces and 27 times its energy."""
    from paper_2001_01583_gb300 import ewald_real_space_forces
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    L, rc, alpha = 9.0, 2.5, 0.8
    r, q = _ions(n, L, "random", n)
    want = ewald.real_space_forces(r, q, L, alpha, rc)
    size = ewald.real_space_energy(r, np.abs(q), L, alpha, rc)
    shifts = L * np.stack(np.meshgrid(*[np.arange(3.0)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    F, got = ewald_real_space_forces(torch.from_numpy((r + shifts).reshape(-1, 3)), torch.from_numpy(np.tile(q, 27)),
                                     3 * L, alpha, rc)
    assert np.abs(F.cpu().numpy().reshape(27, n, 3) - want).max() <= 2e-5 * np.abs(want).max()
    assert abs(got - 27 * ewald.real_space_energy(r, q, L, alpha, rc)) <= 1e-6 * 27 * size
