"""Large decision-only batches filter a frame's combinations in the energy-test stage and mark
them, except those of frames with more combinations than its buffer, which the vertex stage
filters: the decisions equal the plain form's, with both kinds of frame in one warp's share and
with the signal decays that a lost combination would drop."""
import numpy as np
import pytest

from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,light,dense", [(8193, 6.4, 36.0), (8194, 20.0, 34.0), (8197, 34.0, 38.0), (12001, 30.0, 64.0)])
def test_filtered_and_unfiltered_combinations_decide_as_the_plain_form(cfg, n, light, dense):
    from paper_2206_11535_gb300 import m3e
    a, b = gen.generate(n, light, 0.5, 2, seed=700 + n), gen.generate(n // 3 + 1, dense, 0.5, 2, seed=701 + n)
    frames = [a["hits"][a["off"][i]:a["off"][i + 1]] for i in range(n)]
    for k in range(0, n, 3):
        frames[k] = b["hits"][b["off"][k // 3]:b["off"][k // 3 + 1]]
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum([h.size for h in frames])
    h, o = torch.from_numpy(np.concatenate(frames).astype(np.int32)).cuda(), torch.from_numpy(off).cuda()
    with m3e.Context(cfg, 0) as c:
        keep, reason = c.select_frames(h, o)
        want_keep, want_reason = c.select_frames_plain(h, o)
        assert (reason == want_reason).all()
        assert (keep == want_keep).all()
        assert int((reason == m3e.VERTEX).sum()) > 100
