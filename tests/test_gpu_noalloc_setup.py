"""The set-up of m3e_select_frames_noalloc is done by the first call on a device, whatever its
size: after a call of a few frames, a larger one is captured into a graph and replayed."""
import pytest

from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("first", [1, 64, 2048])
def test_a_small_first_call_sets_up_a_captured_larger_one(cfg, first):
    from paper_2206_11535_gb300 import m3e
    n = 4096
    d = gen.generate(n, 10.0, 0.5, 4, seed=first)
    h, o = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    keep, reason = (torch.full((n,), 77, dtype=torch.uint8, device="cuda") for _ in range(2))
    with m3e.Context(cfg, 0) as c:  # a new context forgets the looked-up address
        c.select_frames_noalloc(h, o[:first + 1], keep, reason)
        torch.cuda.synchronize()
        reason.fill_(77)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            c.select_frames_noalloc(h, o, keep, reason)
        assert bool((reason == 77).all())
        g.replay()
        torch.cuda.synchronize()
        want = c.select_frames_plain(h, o)
        assert torch.equal(reason, want[1]) and torch.equal(keep, want[0])
