"""The kernels of a product overlap at their edges, which must not cost more than it gains: a product in a row
of products takes less time than its kernels one by one (each with an event on either side)."""
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


# passes that the FP64 pipe bounds: wide stencils in the gather and the anterpolation, binary64 transforms
@pytest.mark.parametrize("op,s,precision", [("N", 8, 1), ("S_alpha", 4, 2)])
def test_products_in_a_row_take_less_than_their_kernels(aimlib, op, s, precision):
    n = 1000
    ctx = aimlib.Context(synth.StarContour.from_seed(8).polygon(100.0, n), K, aimlib.TE, 230, fft_P=512, s=s, alpha=3.0 * K)
    x = torch.from_numpy(synth.random_coeffs(n, 1, seed=3)).cuda()
    y, count = torch.empty_like(x), 50
    alone = together = math.inf
    for _ in range(5):
        aimlib.profile_start()
        for _ in range(count):
            ctx.matvec(op, x, y, precision=precision)
        torch.cuda.synchronize()
        alone = min(alone, sum(ms for _, ms in aimlib.profile_stop().values()) / count)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(count):
            ctx.matvec(op, x, y, precision=precision)
        e[1].record()
        torch.cuda.synchronize()
        together = min(together, e[0].elapsed_time(e[1]) / count)
    assert together < alone, (together, alone)
    ctx.close()
