"""Row passes at their edges: transform lengths with one and two dense passes behind the sparse
radix, contours whose rows stay below and above the line between the sparse and the dense row pass,
rows along an axis-parallel edge (hundreds of active points, several per residue), and one to nine
right-hand sides (every size of a gather group). Filtered operators need no near field, so the
oracle's FFT product is quick at every size."""
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


CASES = [("star", 3.0, 40, 16, 64), ("star", 6.0, 60, 33, 128), ("square", 6.0, 80, 61, 128),
         ("star", 20.0, 200, 100, 256), ("square", 20.0, 200, 127, 256), ("square", 30.0, 300, 200, 512),
         ("star", 50.0, 300, 400, 1024), ("square", 60.0, 400, 511, 1024), ("square", 100.0, 600, 900, 2048)]


@pytest.mark.parametrize("shape,per,n,m,P", CASES)
def test_filtered_operators_at_row_pass_edges(aimlib, shape, per, n, m, P):
    nodes = square(per / 4.0, n) if shape == "square" else synth.StarContour.from_seed(5).polygon(per, n)
    ctx = aimlib.Context(nodes, K, aimlib.TE, m, fft_P=P, alpha=3.0 * K)
    ref = oaim.TEOperators(nodes, K, m, P, alpha=3.0 * K, L=ctx.info()["L"])
    x = synth.random_coeffs(n, 9, seed=4)
    for op, want in (("S_alpha", ref.S_alpha(x[0])), ("N_alpha", ref.N_alpha(x[0]))):
        for precision in (0, 1, 2):
            saved = ctx.get_schedule(precision)
            for elems in (8, 16):
                try:
                    ctx.set_schedule(precision, 2, 128, 0, elems)
                except aimlib.AimError:
                    continue
                first = None
                for nrhs in (1, 2, 3, 5, 9):
                    xd = torch.from_numpy(x[:nrhs].copy()).cuda()
                    yd = torch.full_like(xd, float("nan"))
                    ctx.matvec(op, xd, yd, precision=precision)
                    y = yd.cpu().numpy()
                    if first is None:
                        first = y[0]
                        err = np.linalg.norm(first - want) / np.linalg.norm(want)
                        assert err < TOL[precision], (op, precision, elems, err)
                    assert np.array_equal(y[0], first), (op, precision, elems, nrhs)
            ctx.set_schedule(precision, **saved)
    ctx.close()
