"""The inverse row pass of full grids: the default launch against the explicit schedules, bit for bit and in
time, at sizes where its transforms per thread used to change."""
import math

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 2.0 * math.pi


@pytest.fixture(scope="module")
def aimlib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10784_gb300 import aim
    return aim


def inverse_time(aim, ctx, u, precision):
    """The product and the microseconds of its inverse row pass, the least of some runs."""
    v, best = torch.empty_like(u), math.inf
    for _ in range(5):
        aim.profile_start()
        for _ in range(5):
            ctx.grid_product(u, v, False, precision=precision)
        torch.cuda.synchronize()
        best = min(best, *[1e3 * ms / count for k, (count, ms) in aim.profile_stop().items() if k.startswith("row_inv")])
    return v, best


@pytest.mark.parametrize("m,P", [(120, 256), (240, 512), (1000, 2048)])
def test_default_launch_is_the_faster_one(aimlib, m, P):
    ctx = aimlib.Context(synth.StarContour.from_seed(3).polygon(5.0, 60), K, aimlib.TE, m, fft_P=P, alpha=2.0 * K)
    u = torch.randn((6 if P == 512 else 1, m, m), dtype=torch.complex128, device="cuda")
    for precision in (0, 1):
        saved = ctx.get_schedule(precision)
        want, took = inverse_time(aimlib, ctx, u, precision)
        for tpt in (1, 2):
            ctx.set_schedule(precision, tpt, 128, 0 if tpt == 1 else 4 if P < 1024 else 2, saved["elems_per_thread"])
            v, other = inverse_time(aimlib, ctx, u, precision)
            assert torch.equal(v, want)
            assert took < 1.1 * other, (precision, tpt, took, other)
        ctx.set_schedule(precision, **saved)
    ctx.close()
