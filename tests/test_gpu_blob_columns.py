"""The last array of a setup blob: which columns of the filtered spectrum the mask of Eq. 10 leaves, read by
builds of the format's first version. It must be in the blob though no context keeps it."""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 2.0 * math.pi


@pytest.mark.parametrize("kw", [dict(alpha=2.0 * K), dict(alpha=8.0 * K), dict(), dict(alpha=2.0 * K, filter_kind=2)])
def test_live_columns_of_a_blob(kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10784_gb300 import aim
    ctx = aim.Context(synth.circle_polygon(2.0, 160), K, aim.TE, 50, **kw)
    info, H = ctx.info(), ctx.info()["fft_P"] // 2
    blob = ctx.export_setup()
    size = (4 * (H + 1) + 15) & ~15
    live = blob[blob.size - size:].view(np.int32)
    kappa = 2.0 * math.pi / (info["fft_P"] * info["eps"]) * np.arange(H + 1)
    want = kappa <= info["alpha"] if info["filter_kind"] == aim.FILTER_NUMERICAL else np.ones(H + 1, bool)
    assert np.array_equal(live[:H + 1], want.astype(np.int32)) and not live[H + 1:].any()
    ctx.close()
