"""Contours that run along the grid: a few grid rows hold many more active points than the others and take
the dense row passes inside a context of sparse rows. Results must not depend on how rows share CTAs, on the
number of right-hand sides or on the kind of launch, and those rows must not set the time of the launch."""
import math

import numpy as np
import pytest

import synth
from oracle import aim as oaim

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 2.0 * math.pi
TOL = {0: 1e-10, 1: 1e-5, 2: 1e-10}      # the operator tolerances of the other parity tests


@pytest.fixture(scope="module")
def aimlib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10784_gb300 import aim
    return aim


def square(side, n):
    """n vertices on an axis-parallel square: its horizontal edges fill whole grid rows."""
    t = 4.0 * np.arange(n) / n
    e, f = np.floor(t).astype(int) % 4, t - np.floor(t)
    x = np.choose(e, [f, np.ones(n), 1.0 - f, np.zeros(n)])
    y = np.choose(e, [np.zeros(n), f, np.ones(n), 1.0 - f])
    return side * np.stack([x - 0.5, y - 0.5], axis=1)


def product(ctx, op, x, precision):
    y = torch.full_like(x, float("nan"))
    ctx.matvec(op, x, y, precision=precision)
    return y


@pytest.mark.parametrize("side,n,m,P", [(5.0, 200, 127, 256), (10.0, 400, 200, 512), (20.0, 800, 400, 1024),
                                        (45.0, 1200, 900, 2048)])
def test_rows_of_both_kinds_in_one_context(aimlib, side, n, m, P):
    nodes = square(side, n)
    ctx = aimlib.Context(nodes, K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
    ref = oaim.TEOperators(nodes, K, m, P, alpha=3.0 * K, L=ctx.info()["L"], near=False)
    x = synth.random_coeffs(n, 3, seed=4)
    xd = torch.from_numpy(x).cuda()
    for op, want in (("S_alpha", ref.S_alpha(x[0])), ("N_alpha", ref.N_alpha(x[0]))):
        for precision, elems in ((0, 8), (0, 16), (1, 8), (1, 16), (2, 16)):
            first = None
            for threads in (32, 128, 512):   # rows per CTA
                ctx.set_schedule(precision, 2, threads, 0, elems)
                y = product(ctx, op, xd, precision)
                if first is None:
                    first = y
                    err = np.linalg.norm(y[0].cpu().numpy() - want) / np.linalg.norm(want)
                    assert err < TOL[precision], (op, precision, elems, err)
                assert torch.equal(y, first), (op, precision, elems, threads)
                assert torch.equal(product(ctx, op, xd[:1].contiguous(), precision)[0], first[0])
            multi = torch.full_like(xd, float("nan"))
            aimlib.matvec_multi([ctx], [op], [xd], [multi], precision=precision)
            assert torch.equal(multi, first), (op, precision, elems)
    ctx.close()


def row_time(aim, ctx, n, precision):
    """Microseconds of the two row passes of S^alpha, the least of some runs."""
    x = torch.from_numpy(synth.random_coeffs(n, 1, seed=3)).cuda()
    y, best = torch.empty_like(x), math.inf
    for _ in range(5):
        aim.profile_start()
        for _ in range(5):
            ctx.matvec("S_alpha", x, y, precision=precision)
        torch.cuda.synchronize()
        t = {k.split()[0]: v for k, v in aim.profile_stop().items()}
        best = min(best, sum(t[k][1] / t[k][0] for k in ("row_fwd", "row_inv")))
    return 1e3 * best


@pytest.mark.parametrize("precision", [0, 1])
def test_long_rows_do_not_set_the_time_of_a_launch(aimlib, precision):
    # the same grid and about the same number of active rows; the square's long rows used to take twice the
    # time of the whole launch of the circle (378 against 165 us in double-float)
    n, m, P = 4000, 2000, 4096
    took = []
    for nodes in (synth.circle_polygon(40.0, n), square(80.0, n)):
        ctx = aimlib.Context(nodes, K, aimlib.TE, m, fft_P=P, alpha=2.0 * K)
        took.append(row_time(aimlib, ctx, n, precision))
        ctx.close()
    assert took[1] < 1.4 * took[0], took


def test_binary64_rows_take_no_longer_than_those_of_a_full_grid(aimlib):
    # a contour of 100 wavelengths: its rows' sums on the FP64 pipe took 109 us where the dense passes take 79
    n, m, P = 1000, 230, 512
    ctx = aimlib.Context(synth.StarContour.from_seed(8).polygon(100.0, n), K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
    u = torch.ones((1, m, m), dtype=torch.complex128, device="cuda")
    v, full = torch.empty_like(u), math.inf
    for _ in range(5):
        aimlib.profile_start()
        for _ in range(5):
            ctx.grid_product(u, v, True, precision=2)
        torch.cuda.synchronize()
        t = {k.split()[0]: w for k, w in aimlib.profile_stop().items()}
        full = min(full, 1e3 * sum(t[k][1] / t[k][0] for k in ("row_fwd", "row_inv")))
    took = row_time(aimlib, ctx, n, 2)
    ctx.close()
    assert took < 1.2 * full, (took, full)


# mean error of six random vectors with every row dense (operators N_alpha, S_alpha), against binary64
DENSE = [(100.0, 1000, 230, 512, 0, 4.43e-14, 1.66e-14), (150.0, 1500, 512, 1024, 0, 6.54e-14, 1.69e-14),
         (400.0, 4000, 1024, 2048, 0, 6.36e-14, 2.03e-14)]


@pytest.mark.parametrize("per,n,m,P,precision,dense_N,dense_S", DENSE)
def test_sparse_rows_are_as_accurate_as_dense_ones(aimlib, per, n, m, P, precision, dense_N, dense_S):
    # a random walk of roundings: the two orders of the same sums differ by a few per cent of their error
    ctx = aimlib.Context(synth.StarContour.from_seed(8).polygon(per, n), K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
    for op, dense in (("N_alpha", dense_N), ("S_alpha", dense_S)):
        errs = []
        for seed in range(6):
            x = torch.from_numpy(synth.random_coeffs(n, 1, seed=seed)).cuda()
            want = product(ctx, op, x, 2)
            errs.append(float((product(ctx, op, x, precision) - want).norm() / want.norm()))
        assert np.mean(errs) < 1.04 * dense, (op, np.mean(errs), dense)
    ctx.close()


# the same for complex64 before radix-8 passes and sparse rows, P = 64 to 2048
DENSE32 = [(5.0, 50, 32, 64, 2.79e-7, 1.72e-7), (12.0, 120, 50, 128, 2.76e-7, 1.71e-7),
           (40.0, 400, 128, 256, 3.18e-7, 1.85e-7), (400.0, 4000, 1024, 2048, 4.02e-7, 2.48e-7)]


@pytest.mark.parametrize("per,n,m,P,dense_N,dense_S", DENSE32)
def test_complex64_is_as_accurate_as_radix_16_passes_of_dense_rows(aimlib, per, n, m, P, dense_N, dense_S):
    test_sparse_rows_are_as_accurate_as_dense_ones(aimlib, per, n, m, P, 1, dense_N, dense_S)
