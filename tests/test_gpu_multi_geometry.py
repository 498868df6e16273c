"""Which schedules may share a multi-context call: contexts that run the same transforms and elements per
thread go together whatever the rest of their schedules says, also where one of them is on the schedule
that contexts of its size start with; each result equals the context's own product bit for bit."""
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


def context(aim, P):
    n, m = P, {256: 120, 512: 200, 2048: 800}[P]
    return aim.Context(synth.StarContour.from_seed(P).polygon(n / 10.0, n), K, aim.TE, m, fft_P=P, alpha=2.0 * K)


# schedules (None: as started) of contexts of the given P, in mixed precision
TOGETHER = [
    [(512, (2, 128, 0, 8)), (512, (2, 256, 0, 8))],
    [(512, (2, 128, 0, 8)), (2048, (2, 128, 0, 8))],
    [(512, None), (2048, (2, 128, 0, 8))],
    [(512, None), (2048, None), (512, (2, 256, 0, 16))],
    [(2048, (2, 128, 0, 0)), (256, None), (2048, (2, 128, 0, 16))],
]
APART = [
    [(512, (2, 256, 0, 8)), (512, (2, 128, 0, 16))],
    [(512, (2, 256, 0, 8)), (2048, None)],
    [(512, None), (512, (2, 256, 0, 8)), (2048, None)],
    [(512, None), (512, (1, 128, 0, 8))],
]


def prepare(aim, specs):
    ctxs = []
    for P, sched in specs:
        c = context(aim, P)
        if sched is not None:
            c.set_schedule(aim.MIXED, *sched)
        ctxs.append(c)
    xs = [torch.from_numpy(synth.random_coeffs(P, 2, seed=i)).cuda() for i, (P, _) in enumerate(specs)]
    return ctxs, xs, [torch.full_like(x, float("nan")) for x in xs]


@pytest.mark.parametrize("specs", TOGETHER)
def test_one_geometry_goes_together(aimlib, specs):
    ctxs, xs, ys = prepare(aimlib, specs)
    aimlib.matvec_multi(ctxs, ["S_alpha"] * len(ctxs), xs, ys, precision=aimlib.MIXED)
    for c, x, y in zip(ctxs, xs, ys):
        want = torch.full_like(x, float("nan"))
        c.matvec("S_alpha", x, want, precision=aimlib.MIXED)
        assert torch.equal(y, want), specs
        c.close()


@pytest.mark.parametrize("specs", APART)
def test_different_geometries_are_refused(aimlib, specs):
    ctxs, xs, ys = prepare(aimlib, specs)
    with pytest.raises(aimlib.AimError) as exc:
        aimlib.matvec_multi(ctxs, ["S_alpha"] * len(ctxs), xs, ys, precision=aimlib.MIXED)
    assert exc.value.status == aimlib.EINVAL and "geometry" in str(exc.value)
    for c in ctxs:
        c.close()
