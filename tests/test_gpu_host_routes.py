"""The host entry point copies and selects batches of at most 8192 frames in order on the
caller's stream, larger ones in chunks: the decisions are the device entry's on both sides of
every line, one call after another on one context and from an offset that does not start at 0."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sizes", [(1, 2048, 2049), (8192, 8193, 5), (12500, 25000, 12499)])
def test_host_entry_decides_as_the_device_entry(cfg, sizes):
    from paper_2206_11535_gb300 import m3e

    from .test_gpu_small_batches import _batch
    with m3e.Context(cfg, 0) as c:
        for n in sizes:
            hits, off = _batch(n)
            want = c.select_frames(torch.from_numpy(hits).cuda(), torch.from_numpy(off).cuda(),
                                   stats=m3e.new_stats())
            h, o = torch.from_numpy(hits).pin_memory(), torch.from_numpy(off).pin_memory()
            cut = min(n - 1, 3)  # a batch that starts inside the buffers
            for a in (0, cut):
                keep, reason = c.select_frames_host(h, o[a:])
                torch.cuda.synchronize()
                assert (reason == want[1].cpu().numpy()[a:]).all()
                assert (keep == want[0].cpu().numpy()[a:]).all()
