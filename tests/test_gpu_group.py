"""The group form (a CTA takes eight frames through the method together) serves
m3e_select_frames_noalloc and middle-sized decision-only batches: its decisions equal the
staged form's (a run with statistics, which always takes it), at whole and ragged groups, at
one wave of CTAs and around it, with frames among them that leave a frame's stage."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2049, 2056, 2063, 4863, 4864, 4865, 8192, 8193, 12000])
def test_group_form_decides_as_the_staged_form(cfg, n):
    from paper_2206_11535_gb300 import m3e

    from .test_gpu_small_batches import _batch
    hits, off = _batch(n)
    h, o = torch.from_numpy(hits).cuda(), torch.from_numpy(off).cuda()
    with m3e.Context(cfg, 0) as c:
        def run(f):
            keep, reason = (torch.full((n,), 77, dtype=torch.uint8, device="cuda") for _ in range(2))
            f(keep, reason)
            torch.cuda.synchronize()
            return keep.cpu().numpy(), reason.cpu().numpy()

        want = run(lambda k, r: c.select_frames(h, o, k, r, stats=m3e.new_stats()))
        got = {"noalloc": run(lambda k, r: c.select_frames_noalloc(h, o, k, r)),
               "noalloc again": run(lambda k, r: c.select_frames_noalloc(h, o, k, r)),
               "select": run(lambda k, r: c.select_frames(h, o, k, r)),
               "graph": run(lambda k, r: c.graph(h, o, k, r).launch())}
        for name, (keep, reason) in got.items():
            assert (reason == want[1]).all(), name
            assert (keep == want[0]).all(), name
