"""An infinite Phi cut has no cosine, and no pair passes the comparison with it: every route finds
no triplet and drops every frame, as the oracle does."""
import copy

import pytest

from oracle import oracle as O
from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cuts", [("phi01_max",), ("phi12_max",), ("phi01_max", "phi12_max")])
def test_no_pair_passes(cfg, cuts):
    from paper_2206_11535_gb300 import m3e
    wide = copy.deepcopy(cfg)
    wide["cuts"].update({k: float("inf") for k in cuts})
    n = 9000
    d = gen.generate(n, 8.0, 0.5, 2, seed=17)
    _, want = O.select_frames(O.make_config(wide), d["hits"], d["off"], 8)
    assert (want == m3e.DROP).all()
    h, o = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    with m3e.Context(wide, 0) as c:
        for k in (1000, 4000, n):
            assert not c.select_frames(h, o[:k + 1])[1].any()
        assert not c.select_frames(h, o, stats=m3e.new_stats())[1].any()
        assert not c.select_frames_plain(h, o)[1].any()
        assert not c.select_frames_fused(h, o)[1].any()
        assert not c.select_frames_noalloc(h, o, *(torch.empty(n, dtype=torch.uint8, device="cuda") for _ in "kr"))[1].any()
        for form in (0, 1, 2):
            assert not c.select_frames_debug(h, o[:501], form=form)["n_trip"].any()
        c.check()
