"""Choices made launch by launch against the explicit ones, at the sizes where they change: passes of one
or two transforms per thread and the column pass of short and long columns (P = 64 to 2048, one to nine
channels), one multi-context call over two pass geometries, Gram rows of the dense and the ring form (127
and 128 unknowns), Krylov cycles around the last step of the one-launch coefficients (128)."""
import math

import numpy as np
import pytest

import synth
from oracle import geometry

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


def uneven(n, seed):
    """n vertices on a smooth contour, neighbouring segments up to a few times longer than one another."""
    rng = np.random.default_rng(seed)
    t = 2.0 * np.pi * (np.arange(n) + rng.uniform(-0.35, 0.35, n)) / n
    r = 1.0 + 0.2 * np.cos(3.0 * t)
    return np.stack([r * np.cos(t), r * np.sin(t)], axis=1)


def product(ctx, op, x, precision):
    y = torch.full_like(x, float("nan"))
    ctx.matvec(op, x, y, precision=precision)
    return y.cpu().numpy()


@pytest.mark.parametrize("per,n,m,P", [(3.0, 40, 24, 64), (20.0, 200, 120, 256), (30.0, 300, 200, 512),
                                       (60.0, 600, 400, 1024), (100.0, 900, 800, 2048)])
def test_default_launches_equal_explicit_schedules(aimlib, per, n, m, P):
    ctx = aimlib.Context(synth.StarContour.from_seed(8).polygon(per, n), K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
    for precision in (0, 1):
        saved = ctx.get_schedule(precision)
        for nrhs in (1, 3):
            x = torch.from_numpy(synth.random_coeffs(n, nrhs, seed=3)).cuda()
            want = {op: product(ctx, op, x, precision) for op in ("N", "S_alpha")}
            for tpt, cols in ((1, 1), (1, 4), (2, 1), (2, 8)):
                try:
                    ctx.set_schedule(precision, tpt, 64, cols, saved["elems_per_thread"])
                except aimlib.AimError:
                    continue
                for op, w in want.items():
                    assert np.array_equal(product(ctx, op, x, precision), w), (op, precision, nrhs, tpt, cols)
            ctx.set_schedule(precision, **saved)
    ctx.close()


def test_multi_context_call_over_two_pass_geometries(aimlib):
    sizes = [(30.0, 300, 200, 512), (100.0, 900, 800, 2048), (60.0, 600, 400, 1024)]
    ctxs = [aimlib.Context(synth.StarContour.from_seed(i).polygon(per, n), K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
            for i, (per, n, m, P) in enumerate(sizes)]
    xs = [torch.from_numpy(synth.random_coeffs(s[1], 2, seed=i)).cuda() for i, s in enumerate(sizes)]
    ops = ["calderon_alpha", "N", "S_alpha"]
    for precision in (0, 1):
        for _ in range(2):   # the second call runs on the buffers the first one left
            ys = [torch.full_like(x, float("nan")) for x in xs]
            aimlib.matvec_multi(ctxs, ops, xs, ys, precision=precision)
            for c, op, x, y in zip(ctxs, ops, xs, ys):
                assert np.array_equal(y.cpu().numpy(), product(c, op, x, precision)), (op, precision)
    ctxs[0].set_schedule(1, 2, 128, 0, 16)   # the geometry of long transforms, named: still one call
    ys = [torch.full_like(x, float("nan")) for x in xs]
    aimlib.matvec_multi(ctxs, ops, xs, ys, precision=1)
    assert np.array_equal(ys[0].cpu().numpy(), product(ctxs[0], ops[0], xs[0], 1))
    ctxs[0].set_schedule(1, 1, 128, 0, 16)
    with pytest.raises(aimlib.AimError) as exc:
        aimlib.matvec_multi(ctxs, ops, xs, ys, precision=1)
    assert exc.value.status == aimlib.EINVAL
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("n", [5, 127, 128, 129, 512, 513])
def test_gram_inverse_on_uneven_meshes(aimlib, n):
    nodes = uneven(n, n)
    ctx = aimlib.Context(nodes, K, aimlib.TE, 64)
    x = synth.random_coeffs(n, 3, seed=n)
    got = product(ctx, "gram_inv", torch.from_numpy(x).cuda(), 0)
    want = np.linalg.solve(geometry.gram_dense(nodes), x.T).T
    # diagonally dominant by a factor of two: the condition is a few times the ratio of the lengths
    assert np.linalg.norm(got - want) < 1e-12 * np.linalg.norm(want)
    ctx.close()


@pytest.mark.parametrize("restart", [127, 128, 129, 300])
def test_solves_around_the_last_one_launch_step(aimlib, restart):
    n, tol = 400, 1e-9
    ctx = aimlib.Context(synth.StarContour.from_seed(6).polygon(40.0, n), K, aimlib.TE, 200, fft_P=512, alpha=3.0 * K)
    b = torch.from_numpy(synth.random_coeffs(n, 2, seed=2)).cuda()
    x = torch.zeros_like(b)
    _, info = ctx.solve("calderon_alpha", b, x, tol=tol, restart=restart, max_iter=restart * 3, precision=0, check=False)
    want = b
    for op in ("gram_inv", "S_alpha", "gram_inv"):
        want = torch.from_numpy(product(ctx, op, want, 0)).cuda()
    want = want.cpu().numpy()
    r = want - product(ctx, "calderon_alpha", x, 0)
    rel = np.linalg.norm(r, axis=1) / np.linalg.norm(want, axis=1)
    for i in range(2):
        assert info[i]["iters"] > 127
        # the solver's residual is the true one up to rounding: 1e-13 of |A| |x|, which exceeds |b| by
        # up to a few thousand in this nearly singular system
        assert abs(rel[i] - info[i]["rel_res"]) < 1e-9, (rel[i], info[i])
        assert not info[i]["converged"] or rel[i] < 2.0 * tol
    ctx.close()


def test_contexts_of_different_shared_memory_take_turns(aimlib):
    # the limit of a kernel's dynamic shared memory is the device's: a context that needs less of it must
    # not take it from one that needs more (147 KB and 74 KB column CTAs of the same kernel)
    ctxs = []
    for per, n, m, P in ((100.0, 900, 800, 2048), (60.0, 600, 400, 1024)):
        c = aimlib.Context(synth.StarContour.from_seed(9).polygon(per, n), K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
        c.set_schedule(0, 2, 128, 4, 8)
        ctxs.append((c, torch.from_numpy(synth.random_coeffs(n, 1, seed=5)).cuda()))
    first = [product(c, "N", x, 0) for c, x in ctxs]
    for _ in range(2):
        for (c, x), want in zip(ctxs, first):
            assert np.array_equal(product(c, "N", x, 0), want)
    for c, _ in ctxs:
        c.close()
