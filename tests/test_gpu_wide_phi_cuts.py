"""Phi cuts above a quarter turn: the thresholds on the scalar product are negative, so a lane
of the warp stage without a layer-1 hit must be kept out by itself.  Every route of a batch
decides as the oracle."""
import copy

import pytest

from oracle import oracle as O
from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("phi01,phi12", [(1.6, 1.6), (2.5, 1.6), (3.1, 3.1), (0.3, 3.1), (3.1, 0.3)])
def test_every_route_decides_as_the_oracle(cfg, phi01, phi12):
    from paper_2206_11535_gb300 import m3e

    from . import parity as P
    wide = copy.deepcopy(cfg)
    wide["cuts"].update(phi01_max=phi01, phi12_max=phi12)
    oc = O.make_config(wide)
    n = 9000
    d = gen.generate(n, 3.0, 0.5, 4, seed=int(100 * phi01 + phi12))
    h, o = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    with m3e.Context(wide, 0) as c:
        rec = {k: v.cpu().numpy() for k, v in c.select_frames_debug(h, o[:301], cap_trip=1024, cap_combo=1024).items()}
        res = P.compare_batch(oc, d["hits"][:d["off"][300]], d["off"][:301], rec)
        assert P.summary(res)["fail"] == 0, [r.fails[:3] for r in res if r.status == "fail"][:5]
        want = c.select_frames_plain(h, o)[1]
        got = {f"first {k}": c.select_frames(h, o[:k + 1])[1] for k in (700, 4000, n)}
        got["statistics"] = c.select_frames(h, o[:4001], stats=m3e.new_stats())[1]
        got["fused"] = c.select_frames_fused(h, o)[1]
        got["noalloc"] = c.select_frames_noalloc(h, o, torch.empty_like(want), torch.empty_like(want))[1]
        for name, r in got.items():
            assert torch.equal(r, want[:r.numel()]), name
        assert int((want == m3e.VERTEX).sum()) > 100
        c.check()
