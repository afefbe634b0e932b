"""The edges of m3e_select_frames and m3e_select_frames_host at batch sizes that reach each of their
routes (a CTA per frame up to 2048 frames, the group form up to 8192, the staged kernels, gated by
the chunks' arrival in the host entry, above): lowered caps, frames that leave a stage of the
group form, batches without hits, invalid addresses, and an autotuned graph."""
import copy

import numpy as np
import pytest

from oracle import oracle as O
from paper_2206_11535_gb300 import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROUTES = [1000, 4000, 9000]


@pytest.fixture(scope="module")
def m3e():
    from paper_2206_11535_gb300 import m3e as mod
    return mod


def _csr(frames):
    off = np.zeros(len(frames) + 1, np.int64)
    off[1:] = np.cumsum([f.size for f in frames])
    return np.concatenate(frames).astype(np.int32), off


def _entries(c, hits, off):
    """The decisions of every decision-only entry point, by name."""
    h, o = torch.from_numpy(hits).cuda(), torch.from_numpy(off).cuda()
    n = off.size - 1
    new = lambda: torch.full((n,), 77, dtype=torch.uint8, device="cuda")  # noqa: E731
    c.prepare(n)
    got = {"select": c.select_frames(h, o, new(), new()), "noalloc": c.select_frames_noalloc(h, o, new(), new())}
    got["graph"] = new(), new()
    g = c.graph(h, o, *got["graph"])
    g.launch()
    keep, reason = np.full(n, 77, np.uint8), np.full(n, 77, np.uint8)
    c.select_frames_host(hits, off, keep, reason)
    torch.cuda.synchronize()
    g.close()
    got = {k: (a.cpu().numpy(), b.cpu().numpy()) for k, (a, b) in got.items()}
    got["host"] = keep, reason
    return got


def _agrees_with_oracle(c, oc, hits, off, reason, want):
    """Every frame as the oracle, but for those whose difference lies in a boundary band."""
    from . import parity as P
    diff = np.nonzero(reason != want)[0]
    assert diff.size <= 0.01 * want.size + 1
    for f in diff:
        h, o = _csr([hits[off[f]:off[f + 1]]])
        rec = {k: v.cpu().numpy() for k, v in
               c.select_frames_debug(torch.from_numpy(h).cuda(), torch.from_numpy(o).cuda(), 1024, 1024).items()}
        assert P.compare_frame(oc, h, P.record_of_frame(rec, 0), int(f)).status == "boundary", int(f)


@pytest.mark.parametrize("n", ROUTES)
def test_lowered_caps(m3e, cfg, n):
    low = copy.deepcopy(cfg)
    low["caps"].update(max_triplets=12, max_tracks=6, max_combos=4)
    oc = O.make_config(low)
    d = gen.workload("c1", n_frames=n, seed=19 + n)
    _, want = O.select_frames(oc, d["hits"], d["off"], 8)
    assert {m3e.DROP, m3e.TRIPLET_OVERFLOW, m3e.TRACK_OVERFLOW, m3e.COMBO_OVERFLOW} <= set(want.tolist())
    with m3e.Context(low, 0) as c:
        got = _entries(c, d["hits"], d["off"])
        _agrees_with_oracle(c, oc, d["hits"], d["off"], got["select"][1], want)
        for name, (keep, reason) in got.items():
            assert (reason == got["select"][1]).all(), name
            assert (keep == (reason != m3e.DROP)).all(), name
        c.check()


def _repeated(n):
    """Frames of at most 160 hits whose layer-1 hits are there two or three times: every triplet, and
    every track of it, as often, so that frames that keep within the group form's hits and
    triplets go beyond its 48 tracks or its 160 combinations."""
    out = []
    for tracks, times, seed in ((8.0, 2, 40), (14.0, 2, 41), (12.0, 3, 42), (16.0, 3, 43)):
        d = gen.generate(n, tracks, 0.0, 2, seed=seed)
        for f in range(n):
            h = d["hits"][d["off"][f]:d["off"][f + 1]]
            more = np.concatenate([h] + [h[(h >> 26) == 1]] * (times - 1))
            if more.size <= 160:
                out.append(more)
    return out


@pytest.mark.parametrize("n", [4000, 9000])
def test_frames_that_leave_the_group_form(m3e, cfg, n):
    pool = _repeated(150)
    light = gen.generate(n, 10.0, 0.5, 2, seed=n)
    frames = [light["hits"][light["off"][i]:light["off"][i + 1]] for i in range(n)]
    for k, h in enumerate(pool):
        frames[3 * k % n] = h
    hits, off = _csr(frames)
    with m3e.Context(cfg, 0) as c:
        h, o = _csr(pool)
        rec = {k: v.cpu().numpy() for k, v in
               c.select_frames_debug(torch.from_numpy(h).cuda(), torch.from_numpy(o).cuda(), 1024, 1024).items()}
        inside = (rec["n_trip"] <= 160) & (np.diff(o) <= 160) & (rec["reason"] != m3e.TRACK_OVERFLOW)
        tracks = ((rec["trk_status"] == 5) & (np.arange(1024) < rec["n_trip"][:, None])).sum(1)
        # combinations that are vertexed in a decision-only run: P_z below the momentum cut
        k = cfg["constants"]["k_MeV_per_T_mm"] * cfg["field"]["B_T"] * cfg["field"]["field_scale"]
        with np.errstate(divide="ignore", invalid="ignore"):
            pz = k / np.abs(rec["trk_val"][..., 0]) * np.cos(rec["trk_val"][..., 1])
        q = rec["combo"][..., :3]
        there = np.arange(1024) < rec["n_combo"][:, None]
        total = np.take_along_axis(pz[:, :, None], np.where(there[..., None], q, 0).reshape(len(pool), -1, 1), 1)
        open_ = (there & (np.abs(total.reshape(len(pool), 1024, 3).sum(2)) < cfg["cuts"]["ptot_max"])).sum(1)
        few = inside & (tracks <= 48) & (rec["reason"] != m3e.COMBO_OVERFLOW)
        assert (inside & (tracks > 48)).sum() > 10 and (few & (open_ > 160)).sum() > 10
        assert (few & (open_ > 0) & (open_ <= 160)).sum() > 10
        want_keep, want = (t.cpu().numpy() for t in c.select_frames_plain(torch.from_numpy(hits).cuda(),
                                                                          torch.from_numpy(off).cuda()))
        for name, (keep, reason) in _entries(c, hits, off).items():
            assert (reason == want).all() and (keep == want_keep).all(), name
        c.check()


@pytest.mark.parametrize("n", ROUTES)
def test_empty_frames_one_frame_and_an_invalid_address(m3e, cfg, n):
    g = cfg["geometry"]
    d = gen.generate(1, 10.0, 0.5, 1, seed=15)
    none, bad = np.zeros(0, np.int32), gen.encode([2], [g["n_ladders"][2]], [0], [0]).astype(np.int32)
    with m3e.Context(cfg, 0) as c:
        for keep, reason in _entries(c, *_csr([none] * n)).values():
            assert (reason == m3e.DROP).all() and (keep == 0).all()
        c.check()
        one = c.select_frames_plain(torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda())[1].item()
        for at in (0, 1, n - 1):
            frames = [none] * n
            frames[at] = d["hits"]
            for keep, reason in _entries(c, *_csr(frames)).values():
                assert reason[at] == one and reason.sum() == one
        c.check()
        for at in (1, n - 1):
            frames = [d["hits"]] * 3 + [none] * (n - 4) + [d["hits"]]
            frames[at] = np.concatenate([frames[at], bad])
            hits, off = _csr(frames)
            want = np.array([one if f.size else 0 for f in frames], np.uint8)
            want[at] = m3e.ERR_BADHIT
            keep, reason = np.full(n, 77, np.uint8), np.full(n, 77, np.uint8)
            c.select_frames_host(hits, off, keep, reason)
            torch.cuda.synchronize()
            assert (reason == want).all() and (keep == (want != 0)).all()
            with pytest.raises(m3e.M3EError) as e:
                c.check()
            assert e.value.code == m3e.EBADHIT
            c.check()
            for keep, reason in _entries(c, hits, off).values():
                assert (reason == want).all() and (keep == (want != 0)).all()
            with pytest.raises(m3e.M3EError):
                c.check()


def test_autotuned_graph_of_the_staged_form(m3e, cfg, ocfg):
    d = gen.workload("c3", n_frames=9000, seed=33)
    _, want = O.select_frames(ocfg, d["hits"], d["off"], 8)
    with m3e.Context(cfg, 0) as c:
        c.autotune(torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda())
        got = _entries(c, d["hits"], d["off"])
        _agrees_with_oracle(c, ocfg, d["hits"], d["off"], got["graph"][1], want)
        for name, (keep, reason) in got.items():
            assert (reason == got["graph"][1]).all() and (keep == (reason != 0)).all(), name
        c.check()


def test_momentum_bound_in_the_staged_form(m3e, cfg):
    d = gen.generate(9000, 10.0, 0.5, 1, seed=71)  # a signal decay in every frame
    h, o = torch.from_numpy(d["hits"]).cuda(), torch.from_numpy(d["off"]).cuda()
    with m3e.Context(cfg, 0) as c:
        want = c.select_frames(h, o, stats=m3e.new_stats())[1].cpu().numpy()
        assert (want == m3e.VERTEX).sum() > 3000
        for name, (_, reason) in _entries(c, d["hits"], d["off"]).items():
            assert (reason == want).all(), name
