"""The two e+ tracks of a combination enter the vertex in an order that their values fix: status,
chi2, target distance and |sum p| of every combination are the same bits whatever the order of a
frame's hits and the numbers that the tracks get from it, in every form."""
import numpy as np
import pytest

from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _combinations(c, hits, off, form):
    """Per frame: {addresses of the e+ pair's and the e-'s hits: [values of each such combination]}."""
    r = c.select_frames_debug(torch.from_numpy(hits).cuda(), torch.from_numpy(off).cuda(), 1024, 1024, form=form)
    r = {k: v.cpu().numpy() for k, v in r.items()}
    out = []
    for f in range(off.size - 1):
        h, got = hits[off[f]:off[f + 1]], {}
        if r["reason"][f] < 2:
            track = [tuple(h[i]) for i in r["trip"][f, :r["n_trip"][f]]]
            for k in range(r["n_combo"][f]):
                a, b, e, status = r["combo"][f, k].tolist()
                pair = tuple(sorted((track[a], track[b])))
                got.setdefault((pair, track[e]), []).append((status, *r["combo_val"][f, k].view(np.int32).tolist()))
        out.append((int(r["reason"][f]), {k: sorted(v) for k, v in got.items()}))
    return out


@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("tracks", [10.0, 20.0])
def test_values_do_not_depend_on_the_hit_order(cfg, form, tracks):
    from paper_2206_11535_gb300 import m3e
    d = gen.generate(400, tracks, 0.5, 1, seed=int(tracks))
    off = d["off"]
    rng = np.random.default_rng(3)
    orders = [np.concatenate([off[f] + np.arange(off[f + 1] - off[f])[::-1] for f in range(400)]),
              np.concatenate([off[f] + rng.permutation(off[f + 1] - off[f]) for f in range(400)])]
    with m3e.Context(cfg, 0) as c:
        want = _combinations(c, d["hits"], off, form)
        assert sum(len(v) for _, v in want) > 2000
        for o in orders:
            assert _combinations(c, np.ascontiguousarray(d["hits"][o]), off, form) == want
