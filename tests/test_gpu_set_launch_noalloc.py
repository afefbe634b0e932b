"""m3e_set_launch limits the resident CTAs of m3e_select_frames_noalloc: with one CTA per SM
instead of four a batch of many groups takes clearly longer, and its decisions stay."""
import pytest

from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_ctas_per_sm_reaches_noalloc(cfg):
    from paper_2206_11535_gb300 import m3e
    d = gen.generate(50_000, 6.4, 0.5, 10, seed=9)
    h, o = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    keep, reason = (torch.empty(50_000, dtype=torch.uint8, device="cuda") for _ in range(2))
    with m3e.Context(cfg, 0) as c:
        want = c.select_frames_plain(h, o)

        def run(ctas):
            c.set_launch(4, ctas)
            ms = []
            for _ in range(8):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                c.select_frames_noalloc(h, o, keep, reason)
                b.record()
                torch.cuda.synchronize()
                assert torch.equal(keep, want[0]) and torch.equal(reason, want[1])
                ms.append(a.elapsed_time(b))
            return min(ms)

        assert run(1) > 1.5 * run(0) and run(4) < 1.2 * run(0)
