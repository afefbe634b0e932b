"""A geometry whose look-up tables do not fit an SM's shared memory: the ingest gives the same
coordinates on both sides of the line between its kernels, where a context of that geometry exists."""
import copy

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_rows", [8192, 2048])
@pytest.mark.parametrize("phi", [True, False])
def test_large_tables_are_ingested_at_every_size(cfg, n_rows, phi):
    from paper_2206_11535_gb300 import m3e
    big = copy.deepcopy(cfg)
    big["geometry"].update(n_ladders=[32] * 4, n_cols=[256] * 4, n_rows=[n_rows] * 4)
    g = torch.Generator(device="cuda").manual_seed(n_rows)
    n = 2_000_003
    r = lambda v: torch.randint(v, (n,), generator=g, device="cuda")  # noqa: E731
    h = ((r(4) << 26) | (r(32) << 21) | (r(256) << 13) | r(n_rows)).int()
    with m3e.Context(big, 0) as c:
        got = c.ingest(h, with_phi=phi)
        parts = [c.ingest(h[a:b], with_phi=phi) for a, b in ((0, 1_000_000), (1_000_000, n))]
        for k in range(4 if phi else 3):
            want = torch.cat([p[k] for p in parts])
            assert torch.equal(got[k].view(torch.int32), want.view(torch.int32))
        c.check()
    L, col, row = (h >> 26).long(), ((h >> 13) & 8191).double(), (h & 8191).double()
    geo = big["geometry"]
    at = lambda v: torch.tensor(v, device="cuda", dtype=torch.float64)[L]  # noqa: E731
    ph = (col + 0.5) * (2 * torch.pi / 8192)
    # one rounding to FP32 of values below 128 mm and 1024 mm
    assert (got[0].double() - at(geo["r_mm"]) * torch.cos(ph)).abs().max() < 4e-6
    assert (got[1].double() - at(geo["r_mm"]) * torch.sin(ph)).abs().max() < 4e-6
    assert (got[2].double() - ((row + 0.5) * geo["pitch_mm"] - at(geo["half_len_mm"]))).abs().max() < 3.06e-5
