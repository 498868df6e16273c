"""G^-1 entry by entry where its rows are stored whole (up to 512 unknowns): its columns against an elimination
in 80 digits, also where they are far below the rounding of the diagonal, and a value that is not finite, which
must reach every unknown."""
import math
from decimal import Decimal, getcontext

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


def inverse_column(G, col):
    """Column `col` of the inverse of a cyclic tridiagonal matrix: elimination from unknown 0 on, which carries
    the last column along."""
    getcontext().prec = 80
    n = len(G)
    D = lambda i, j: Decimal(float(G[i % n, j % n]))
    diag, last, rhs = [None] * n, [None] * n, [Decimal(0)] * n
    rhs[col] = Decimal(1)
    diag[0], last[0] = D(0, 0), D(0, n - 1)
    corner, corner_diag, corner_rhs = D(n - 1, 0), D(n - 1, n - 1), rhs[n - 1]
    for i in range(n - 2):       # row i: diag x_i + D(i, i + 1) x_{i+1} + last x_{n-1} = rhs
        f = corner / diag[i]
        corner_diag, corner_rhs = corner_diag - f * last[i], corner_rhs - f * rhs[i]
        corner = (D(n - 1, n - 2) if i == n - 3 else Decimal(0)) - f * D(i, i + 1)
        f = D(i + 1, i) / diag[i]
        diag[i + 1] = D(i + 1, i + 1) - f * D(i, i + 1)
        last[i + 1] = (D(n - 2, n - 1) if i == n - 3 else Decimal(0)) - f * last[i]
        rhs[i + 1] = rhs[i + 1] - f * rhs[i]
    f = corner / diag[n - 2]
    x = [Decimal(0)] * n
    x[n - 1] = (corner_rhs - f * rhs[n - 2]) / (corner_diag - f * last[n - 2])
    x[n - 2] = (rhs[n - 2] - last[n - 2] * x[n - 1]) / diag[n - 2]
    for i in range(n - 3, -1, -1):
        x[i] = (rhs[i] - D(i, i + 1) * x[i + 1] - last[i] * x[n - 1]) / diag[i]
    return np.array([float(v) for v in x])


@pytest.mark.parametrize("n", [128, 129, 300, 512])
def test_every_entry_of_a_column(aimlib, n):
    nodes = synth.StarContour.from_seed(n).polygon(n / 10.0, n)
    ctx = aimlib.Context(nodes, K, aimlib.TE, 64)
    G = geometry.gram_dense(nodes)
    for col in (0, n // 3):
        x = torch.zeros((1, n), dtype=torch.complex128, device="cuda")
        x[0, col] = 1.0
        y = torch.full_like(x, float("nan"))
        ctx.matvec("gram_inv", x, y)
        want = inverse_column(G, col)
        # a product of up to n ratios of a few roundings each
        assert np.max(np.abs(y[0].cpu().numpy().real - want) / np.abs(want)) < 8.0 * n * 2.0 ** -53
    x[0, 0] = float("nan")
    ctx.matvec("gram_inv", x, y)
    assert torch.isnan(y.real).all()
    ctx.close()
