"""The two ingest kernels (look-ups from global memory up to 2,000,000 hits, from shared memory
above) and their reads of unaligned sub-ranges give the same bits, at the sizes around the line
and at ragged ends; an invalid address in the last hit is seen by every route."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LINE = 2_000_000


@pytest.fixture(scope="module")
def hits(cfg):
    g = torch.Generator(device="cuda").manual_seed(7)
    n = LINE + 4096
    geo = cfg["geometry"]
    L = torch.randint(4, (n,), generator=g, device="cuda")
    pick = lambda v: (torch.rand(n, generator=g, device="cuda") * torch.tensor(v, device="cuda")[L]).long()  # noqa: E731
    lad, col, row = pick(geo["n_ladders"]), pick(geo["n_cols"]), pick(geo["n_rows"])
    return ((L << 26) | (lad << 21) | (col << 13) | row).int()


@pytest.mark.parametrize("skip", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [LINE - 1, LINE, LINE + 1, LINE + 2, LINE + 3, LINE + 4])
@pytest.mark.parametrize("phi", [True, False])
def test_routes_agree(cfg, hits, n, skip, phi):
    from paper_2206_11535_gb300 import m3e
    with m3e.Context(cfg, 0) as c:
        h = hits[skip:skip + n].clone() if skip == 0 else hits[skip:skip + n]
        got = c.ingest(h, with_phi=phi)
        # pieces of the same batch, each through the other kernel or another alignment
        cut = 999_937
        parts = [c.ingest(h[a:b], with_phi=phi) for a, b in ((0, cut), (cut, n))]
        for k in range(4 if phi else 3):
            want = torch.cat([p[k] for p in parts])
            assert torch.equal(got[k].view(torch.int32), want.view(torch.int32))
        c.check()
        bad = h.clone()
        bad[n - 1] = -1
        x = c.ingest(bad, with_phi=phi)[0]
        assert torch.isnan(x[n - 1]) and torch.equal(x[:n - 1], got[0][:n - 1])
        with pytest.raises(m3e.M3EError):
            c.check()
