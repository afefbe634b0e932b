"""Small batches take a CTA per frame: their decisions equal the staged form's (a run with
statistics, which always takes it) and the plain form's, at the sizes where the kernel's
variant or the route changes, with frames that the small stage cannot hold among them."""
import numpy as np
import pytest

from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _batch(n):
    """n frames: the parity mix, with every kind of frame that leaves the small stage spread over it."""
    light = gen.generate(n, 10.0, 0.5, 4, seed=90 + n)
    dense = gen.generate(24, 75.0, 0.5, 4, seed=91)          # above 512 triplets or max_triplets
    noisy = gen.generate(6, 5.0, 150.0, None, seed=92)       # above 512 hits
    huge = gen.generate(2, 5.0, 1100.0, None, seed=93)       # above max_hits
    odd = [np.zeros(0, np.int32), np.array([-1], np.int32), dense["hits"][:dense["off"][1]].copy()]
    odd[2][3] = (1 << 26) | 8191                             # a row that the layer does not have
    pool = [d["hits"][d["off"][i]:d["off"][i + 1]] for d in (dense, noisy, huge) for i in range(d["off"].size - 1)] + odd
    frames = [light["hits"][light["off"][i]:light["off"][i + 1]] for i in range(n)]
    for k, h in enumerate(pool):
        if n > 1:
            frames[(k * 61 + 7) % n] = h
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum([h.size for h in frames])
    return np.concatenate(frames).astype(np.int32), off


@pytest.mark.parametrize("n", [1, 3, 152, 607, 608, 609, 2047, 2048, 2049])
def test_small_batches_decide_as_the_staged_form(cfg, n):
    from paper_2206_11535_gb300 import m3e
    hits, off = _batch(n)
    h, o = torch.from_numpy(hits).cuda(), torch.from_numpy(off).cuda()
    with m3e.Context(cfg, 0) as c:
        def run(f):
            keep, reason = (torch.full((n,), 77, dtype=torch.uint8, device="cuda") for _ in range(2))
            f(keep, reason)
            torch.cuda.synchronize()
            return keep.cpu().numpy(), reason.cpu().numpy()

        want = run(lambda k, r: c.select_frames(h, o, k, r, stats=m3e.new_stats()))
        c.prepare(n)
        got = {"small": run(lambda k, r: c.select_frames(h, o, k, r)),
               "again": run(lambda k, r: c.select_frames(h, o, k, r)),
               "plain": run(lambda k, r: c.select_frames_plain(h, o, k, r)),
               "noalloc": run(lambda k, r: c.select_frames_noalloc(h, o, k, r)),
               "graph": run(lambda k, r: c.graph(h, o, k, r).launch())}
        for name, (keep, reason) in got.items():
            assert (reason == want[1]).all(), name
            assert (keep == want[0]).all(), name
        if n > 100:
            assert {m3e.VERTEX, m3e.TRIPLET_OVERFLOW, m3e.HIT_OVERFLOW, m3e.ERR_BADHIT} <= set(want[1].tolist())
            with pytest.raises(m3e.M3EError):
                c.check()
