"""Transforms captured into CUDA graphs before the plan's first forces call give the same results when they are replayed
after it: the forces keep to buffers of their own, and the plan's grid stays where the graphs have it.  The forces'
call is captured as well (its buffers exist from the call before).

Bars: the transforms and forces of two runs differ by the order of FP32 (FP64) atomic sums only: 1e-5 (1e-12) of the rms.
"""
import numpy as np
import pytest

from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("capacity", [1, 2, 3])
def test_captured_transforms_after_forces(precision, tol, capacity):
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N, M, L, alpha = (16, 12, 18), 2000, 10.0, 0.8
    dt = torch.complex128 if precision == "fp64" else torch.complex64
    x = torch.from_numpy(inputs.uniform_points(M, 3, seed=3)).cuda()
    q = torch.from_numpy(np.random.default_rng(4).choice([-1.0, 1.0], M)).to(dt).cuda()
    f = torch.from_numpy(inputs.complex_normal(M, seed=5)).to(dt).cuda()
    fh = torch.from_numpy(inputs.complex_normal(N, seed=6)).to(dt).cuda()
    a, b = torch.empty(N, dtype=dt, device="cuda"), torch.empty(M, dtype=dt, device="cuda")
    F = torch.empty((M, 3), dtype=torch.float64, device="cuda")

    def close(got, want):
        assert float((got - want).abs().max()) <= tol * float(want.abs().square().mean().sqrt())

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream), Plan(N, M, 2.0, 4, "kaiser_bessel", precision) as p:
        if capacity > 1:
            p.set_option(_lib.OPT_RHS_CAPACITY, capacity)
        p.set_points(x)
        want_a, want_b = p.adjoint(f).clone(), p.forward(fh).clone()
        p.sync()
        transforms = torch.cuda.CUDAGraph()
        with torch.cuda.graph(transforms, stream=stream):
            p.adjoint(f, a)
            p.forward(fh, b)
        want_F = p.ewald_reciprocal_forces(q, L, alpha).clone()
        p.sync()
        # what the forces call may have freed, if anything, is written over
        spare = [torch.full((1 << 20,), 7.0, device="cuda") for _ in range(8)]
        a.zero_()
        b.zero_()
        transforms.replay()
        p.sync()
        close(a, want_a)
        close(b, want_b)
        forces = torch.cuda.CUDAGraph()
        with torch.cuda.graph(forces, stream=stream):
            p.ewald_reciprocal_forces(q, L, alpha, F)
        F.zero_()
        forces.replay()
        p.sync()
        close(F, want_F)
        close(p.adjoint(f), want_a)
        del spare
