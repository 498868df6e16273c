"""A multi-context launch whose grid barrier gives up: what it leaves behind is set from the host (no launch
is made to hang), and the calls that follow must report it once and then work again."""
import ctypes
import math
import os
import subprocess
import threading
import time

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 2.0 * math.pi
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def aimlib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10784_gb300 import aim
    return aim


@pytest.fixture(scope="module")
def probe(aimlib, tmp_path_factory):
    out = str(tmp_path_factory.mktemp("probe") / "probe.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(os.path.dirname(aimlib.LIB_PATH), "csrc"),
                    "-I", os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
                    os.path.join(HERE, "multi_launcher_probe.cpp"), "-o", out], check=True, timeout=120)
    ctypes.CDLL(aimlib.LIB_PATH, mode=ctypes.RTLD_GLOBAL)
    lib = ctypes.CDLL(out)
    flags = ctypes.POINTER(ctypes.c_int)
    for f, t in ((lib.probe_err_host, flags), (lib.probe_scratch, ctypes.c_void_p), (lib.probe_batcher_err_host, flags)):
        f.argtypes, f.restype = [ctypes.c_void_p], t
    return lib


class Words:
    """`count` 32-bit words at a device address, for torch."""

    def __init__(self, address, count):
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": "<i4", "data": (address, False), "version": 2}


def give_up(err_host, scratch, stage):
    """The state that a launch of `stage` leaves when a wait gives up: arrivals of CTAs that left, error flags."""
    words = torch.as_tensor(Words(scratch + 16 * stage, 4), device="cuda")
    words.copy_(torch.tensor([3, 0, 1, 0], dtype=torch.int32))
    torch.cuda.synchronize()
    err_host[stage] = 1


def contexts(aim, sizes):
    return [aim.Context(synth.StarContour.from_seed(i).polygon(n / 10.0, n), K, aim.TE, m, alpha=2.0 * K)
            for i, (n, m) in enumerate(sizes)]


def vectors(sizes, nrhs=2):
    return [torch.from_numpy(synth.random_coeffs(n, nrhs, seed=i)).cuda() for i, (n, _) in enumerate(sizes)]


@pytest.mark.parametrize("stage", [0, 1])
def test_a_failed_call_leaves_nothing_to_the_next(aimlib, probe, stage):
    sizes = [(60, 32), (150, 64)]
    ctxs, xs = contexts(aimlib, sizes), vectors(sizes)
    ys = [torch.empty_like(x) for x in xs]
    ops = ["calderon_alpha"] * 2
    aimlib.matvec_multi(ctxs, ops, xs, ys)
    want = [y.clone() for y in ys]
    # a give-up alone: reported by its own call, and by no other
    give_up(probe.probe_err_host(ctxs[0]._h), probe.probe_scratch(ctxs[0]._h), stage)
    with pytest.raises(aimlib.AimError) as exc:
        aimlib.matvec_multi(ctxs, ops, xs, ys)
    assert exc.value.status == aimlib.ETIMEOUT
    aimlib.matvec_multi(ctxs, ops, xs, ys)
    assert all(torch.equal(y, w) for y, w in zip(ys, want))
    # a give-up in a call that fails for another reason: that reason is reported, and the next call works
    give_up(probe.probe_err_host(ctxs[0]._h), probe.probe_scratch(ctxs[0]._h), stage)
    with pytest.raises(aimlib.AimError) as exc:
        aimlib.matvec_multi(ctxs, ["calderon_alpha", "efie_alpha"], xs, ys)
    assert exc.value.status == aimlib.ESTATE
    for y in ys:
        y.fill_(float("nan"))
    aimlib.matvec_multi(ctxs, ops, xs, ys)
    assert all(torch.equal(y, w) for y, w in zip(ys, want))
    for c in ctxs:
        c.close()


def test_a_second_init_takes_up_the_pinned_flags(probe):
    assert probe.probe_init_keeps_flags() == 1


def solve(aim, ctx, batcher, out, i, max_iter):
    n = ctx.n
    b = torch.from_numpy(synth.random_coeffs(n, 1, seed=i)).cuda()
    x, st = torch.zeros_like(b), torch.cuda.Stream()
    torch.cuda.synchronize()
    out[i] = ctx.solve("calderon", b, x, tol=1e-15, restart=60, max_iter=max_iter, stream=st, check=False,
                       batcher=batcher)[0]


def test_a_batcher_that_gave_up_refuses_and_reports(aimlib, probe):
    sizes = [(150, 64), (160, 64), (1100, 300)]   # P = 128 twice, and P = 1024, which is not fused
    ctxs, out = contexts(aimlib, sizes), {}
    batcher = aimlib.Batcher(max_wait_us=100)
    # the first solve runs for many seconds if nothing stops it; the flag is raised while it keeps the stream busy
    t = threading.Thread(target=solve, args=(aimlib, ctxs[0], batcher, out, 0, 200000))
    t.start()
    while batcher.stats()["launches"] < 50:
        assert t.is_alive()
        time.sleep(0.01)
    probe.probe_batcher_err_host(batcher._h)[1] = 1
    solve(aimlib, ctxs[1], batcher, out, 1, 40)
    t.join(timeout=60)
    assert not t.is_alive()
    assert out == {0: aimlib.ETIMEOUT, 1: aimlib.ETIMEOUT}
    # nothing is launched any more, and a solve that never fuses is not concerned
    before = batcher.stats()["launches"]
    solve(aimlib, ctxs[1], batcher, out, 1, 40)
    solve(aimlib, ctxs[2], batcher, out, 2, 40)
    assert out[1] == aimlib.ETIMEOUT and out[2] == aimlib.ENOCONV
    assert batcher.stats()["launches"] == before
    batcher.close()
    for c in ctxs:
        c.close()
