"""m3e_autotune puts only a number of frames per grab in force that ran on the calibration batch,
or leaves the setting that it found: a batch runs with at most one frame per grab for every two
grabs of a resident warp, so a small one says nothing about the larger numbers."""
import pytest

from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,grab", [(3000, 4), (3000, 16), (60_000, 4), (200_000, 64)])
def test_grabs_in_force_have_run(cfg, n, grab):
    from paper_2206_11535_gb300 import m3e
    d = gen.generate(n, 6.4, 0.5, 10, seed=n)
    h, o = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with m3e.Context(cfg, 0) as c:
        c.set_launch(grab)
        t = c.autotune(h, o)
        most = max(1, n // (2 * 4 * sms * t["s1_ctas_per_sm"]))  # 4 warps of a CTA
        assert t["frames_per_grab"] == grab or t["frames_per_grab"] <= most
        # each number that runs is timed once: of 3000 frames one, with 3 hit limits and 2 CTA
        # counts, beside the default and at most 6 settings of the other axes
        if n == 3000:
            assert t["configs_tried"] <= 1 + 6 + 6
        assert torch.equal(c.select_frames(h, o)[1], c.select_frames_plain(h, o)[1])
