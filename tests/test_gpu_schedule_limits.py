"""Exactly the schedules that fit a CTA are accepted: at least a warp and at most the launch bound of threads,
two padded transforms of each of its lines in 227 KB of shared memory, and in binary64 two transforms of 16
elements per thread only."""
import math

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 2.0 * math.pi


def fits(precision, P, tpt, cols, elems):
    H, size = P // 2, 8 if precision == 1 else 16
    if precision == 2 and (tpt, elems) != (2, 16):
        return False
    bound = min(1024, (1024 if precision == 1 else 512) // tpt * (16 // elems))
    per_line = (3 - tpt) * H // elems
    padded = H + H // elems + 2
    return (H >= 2 * elems and 32 <= cols * per_line <= bound and per_line <= bound
            and 2 * cols * padded * size <= 227 * 1024)


@pytest.mark.parametrize("m,P", [(24, 64), (50, 128), (120, 256), (200, 512), (400, 1024), (800, 2048), (1500, 4096)])
def test_accepted_schedules(m, P):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10784_gb300 import aim
    ctx = aim.Context(synth.StarContour.from_seed(1).polygon(5.0, 60), K, aim.TE, m, fft_P=P)
    accepted = 0
    for precision in (0, 1, 2):
        saved = ctx.get_schedule(precision)
        for tpt in (1, 2):
            for elems in (8, 16):
                for cols in (1, 2, 4, 8, 16):
                    try:
                        ctx.set_schedule(precision, tpt, 128, cols, elems)
                        ok = True
                    except aim.AimError as e:
                        assert e.status == aim.EINVAL
                        ok = False
                    assert ok == fits(precision, P, tpt, cols, elems), (precision, tpt, cols, elems)
                    accepted += ok
        ctx.set_schedule(precision, **saved)
        ctx.set_schedule(precision, 2, 128, 0, 16)   # the default columns fit at every length
    assert accepted >= 15
    ctx.close()
