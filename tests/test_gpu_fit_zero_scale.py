"""At a field scale of 0 no candidate has a fit: the sum, its gradient and the count are 0."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("scale", [0.0, -0.0])
def test_zero_field_scale_gives_zero(cfg, scale):
    from paper_2206_11535_gb300 import m3e
    d = gen.generate(100, 10.0, 0.5, 4, seed=5)
    hits, off = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    p = torch.tensor(np.asarray(O.nominal_params()), dtype=torch.float32, device="cuda")
    with m3e.Context(cfg, 0) as c:
        rec = {k: v.cpu().numpy() for k, v in c.select_frames_debug(hits, off).items()}
        cand = torch.from_numpy(m3e.kept_candidates(rec, d["off"])).cuda()
        assert cand.shape[0] > 100
        p[24] = scale
        s, g = c.fit_grad(hits, off, cand, p)
        assert s.item() == 0.0 and torch.count_nonzero(g).item() == 0 and not torch.isnan(g).any()
        assert c.fit_valid_count() == 0
