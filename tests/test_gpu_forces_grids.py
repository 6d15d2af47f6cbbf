"""The forces' three grids: a plan that has computed forces goes on giving the same transforms, before and after its
right-hand-side capacity changes, and the same forces again (small grids: three at once; a grid above the limit: one
after another)."""
import numpy as np
import pytest

from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision,tol", [((16, 12, 18), "fp64", 1e-12), ((16, 12, 18), "fp32", 1e-5),
                                             ((100, 96, 90), "fp32", 1e-5)])
def test_transforms_around_forces(N, precision, tol):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    M, L, dt = 2000, 10.0, torch.complex128 if precision == "fp64" else torch.complex64
    x = torch.from_numpy(inputs.uniform_points(M, 3, seed=3)).cuda()
    q = torch.from_numpy(np.random.default_rng(4).choice([-1.0, 1.0], M)).to(dt).cuda()
    f = torch.from_numpy(inputs.complex_normal((2, M), seed=5)).to(dt).cuda()

    def close(a, b):
        assert float((a - b).abs().max()) <= tol * float(b.abs().square().mean().sqrt())

    with Plan(N, M, 2.0, 4, "kaiser_bessel", precision) as p:
        p.set_points(x)
        a = p.adjoint(f)
        b = p.forward(a)
        F = p.ewald_reciprocal_forces(q, L, 0.8)
        close(p.adjoint(f), a)
        close(p.forward(a), b)
        assert p.info()["rhs_capacity"] == 1
        close(p.ewald_reciprocal_forces(q, L, 0.8), F)
        p.set_option(_lib.OPT_RHS_CAPACITY, 2)
        p.set_points(x)
        close(p.forward(a), b)
        close(p.ewald_reciprocal_forces(q, L, 0.8), F)
        close(p.adjoint(f), a)
        p.sync()
