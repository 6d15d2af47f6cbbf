"""Pencils have blocks of their own: the thread options leave them as they are, and the autotuner times no thread counts for
a plan of pencils only."""
import pytest

from paper_2001_01583_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_autotune_times_no_thread_counts_for_pencils():
    from paper_2001_01583_gb300 import Plan
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N, M = (32, 32, 32), 200000
    with Plan(N, M, 2.0, 4, "kaiser_bessel", "fp32") as p:
        p.set_points(torch.from_numpy(inputs.uniform_points(M, 3, seed=1)).cuda())
        p.autotune(2)
        info = p.info()
    assert info["bin"][0] != 1023 or info["spread_threads"] == info["interp_threads"] == 0


def test_thread_options_leave_pencils_alone():
    from paper_2001_01583_gb300 import Plan, _lib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N, M = (16, 16, 16), 20000
    x = torch.from_numpy(inputs.uniform_points(M, 3, seed=1)).cuda()
    f = torch.from_numpy(inputs.complex_normal(M, seed=2)).to(torch.complex64).cuda()
    with Plan(N, M, 2.0, 4, "kaiser_bessel", "fp32") as p:
        p.set_points(x)
        a = p.adjoint(f)
        blocks = p.info()["spread_block_threads"]
        for option in (_lib.OPT_THREADS, _lib.OPT_SPREAD_THREADS, _lib.OPT_INTERP_THREADS):
            p.set_option(option, 64)
        b = p.adjoint(f)
        p.sync()
        assert p.info()["spread_block_threads"] == blocks
        assert float((a - b).abs().max()) <= 1e-5 * float(a.abs().square().mean().sqrt())
