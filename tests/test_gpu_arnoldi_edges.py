"""Krylov cycles that end at the last steps of the one-launch coefficients and at the first of the three-launch
ones (128 steps), against the oracle's GMRES: the residual and the solution after exactly that many steps, on a
system whose residual falls by half in every step there, so that a wrong last column shows."""
import math

import numpy as np
import pytest

import synth
from oracle import aim as oaim, solve as osolve

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 2.0 * math.pi
N, M, P = 400, 96, 256


@pytest.fixture(scope="module")
def system():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10784_gb300 import aim
    nodes = synth.StarContour.from_seed(6).polygon(40.0, N)
    ctx = aim.Context(nodes, K, aim.TE, M, fft_P=P, alpha=2.0 * K)
    A = osolve.assemble(oaim.TEOperators(nodes, K, M, P, alpha=2.0 * K, L=ctx.info()["L"]).N, N)
    yield ctx, A, synth.random_coeffs(N, 2, seed=2)
    ctx.close()


def solve(ctx, b, **kw):
    bd = torch.from_numpy(b).cuda()
    x = torch.zeros_like(bd)
    _, info = ctx.solve("efie", bd, x, precision=0, check=False, **kw)
    return x.cpu().numpy(), info


@pytest.mark.parametrize("steps", [1, 2, 126, 127, 128, 129, 130])
def test_a_cycle_of_exactly_this_many_steps(system, steps):
    # perturbing A by 1e-12 changes these residuals by up to 4e-5 and the solutions by 6e-12; the operators agree
    # to 1e-10 at worst and to 1e-13 in use
    ctx, A, b = system
    x, info = solve(ctx, b, tol=1e-14, restart=steps, max_iter=steps)
    for r in range(2):
        want, iters, _ = osolve.gmres(lambda v: A @ v, b[r], tol=1e-14, restart=steps, max_iter=steps)
        res = np.linalg.norm(b[r] - A @ want) / np.linalg.norm(b[r])
        assert info[r]["iters"] == iters == steps
        assert abs(info[r]["rel_res"] / res - 1.0) < 1e-3, (info[r], res)
        assert np.linalg.norm(x[r] - want) < 1e-9 * np.linalg.norm(want)


@pytest.mark.parametrize("restart", [127, 128, 300])
def test_iterations_of_a_whole_solve(system, restart):
    ctx, A, b = system
    x, info = solve(ctx, b, tol=1e-12, restart=restart, max_iter=400)
    for r in range(2):
        _, iters, _ = osolve.gmres(lambda v: A @ v, b[r], tol=1e-12, restart=restart, max_iter=400)
        assert info[r]["converged"] and abs(info[r]["iters"] - iters) <= 1, (info[r], iters)
        assert np.linalg.norm(b[r] - A @ x[r]) < 1e-10 * np.linalg.norm(b[r])
