"""Performance cases of the library: what its users have it do, through its public entry points.

Frames are drawn on the GPU from the detector model of the repository's generator (helices from
the hollow double-cone target through the four pixel layers, Highland scattering, digitisation,
uniform noise, three-track signal decays), because a batch of a million frames takes minutes on
the host.  The mixes are those of the benchmark and the tests: the paper's nominal muon rate
(6.4 tracks, 0.5 noise hits per layer), the parity mix (10 tracks, 0.5), the throughput mix (20
tracks, 2), uneven frames (lognormal track counts, one frame in a hundred with 100 times the
noise) and the higher muon rates (32 and 64 tracks).

Kinds of case:
  select   Context.select_frames on device buffers
  graph    the same batch captured once and launched as a CUDA graph
  host     Context.select_frames_host from page-locked host buffers
  noalloc  Context.select_frames_noalloc, for loops that may not allocate
  ingest   Context.ingest: addresses to x, y, z, phi
  align    one step of an alignment fit: fit_chi2_sum forward and backward
  grad     Context.fit_grad alone
  each     Context.fit_chi2 and Context.fit_kappa of every candidate
"""
import math

import numpy as np
import torch

from paper_2206_11535_gb300 import gen, m3e

TWO_PI = 2.0 * math.pi
CHUNK = 1 << 17  # frames drawn at a time


def _select(kind, frames, tracks, noise, signal_every, uneven=False):
    return {"kind": kind, "frames": frames, "tracks": tracks, "noise": noise, "signal_every": signal_every,
            "uneven": uneven}


def listed():
    return [
        # a hand-off of a few microseconds of data at the nominal rate: launches and latency
        {"name": "select_64", **_select("select", 64, 6.4, 0.5, 10)},
        # the parity batch: an ordinary small call
        {"name": "select_1000", **_select("select", 1000, 10.0, 0.5, 10)},
        # offline reprocessing: the benchmark's throughput batch
        {"name": "select_1m", **_select("select", 1_000_000, 20.0, 2.0, 1000)},
        # uneven frames, the benchmark's persistent batched form
        {"name": "graph_uneven", **_select("graph", 200_000, 15.0, 0.5, 1000, True)},
        # five times the nominal muon rate, an odd number of frames
        {"name": "select_dense", **_select("select", 20_001, 32.0, 0.5, 1000)},
        # end to end from host memory, as a filter process receives its data
        {"name": "host_200k", **_select("host", 200_000, 20.0, 2.0, 1000)},
        # one millisecond of 64 ns frames in a fixed-rate loop
        {"name": "noalloc_1ms", **_select("noalloc", 15_625, 6.4, 0.5, 1000)},
        # decoded coordinates of the throughput batch's hits, and of a small odd number of hits
        {"name": "ingest_85m", "kind": "ingest", "hits": 85_500_000, "skip": 0, "phi": True},
        {"name": "ingest_30k", "kind": "ingest", "hits": 30_011, "skip": 0, "phi": True},
        # one optimiser step over the alignment sample's candidates
        {"name": "align_970k", "kind": "align", "candidates": 971_437},
        # the gradient over a small monitoring sample
        {"name": "grad_5k", "kind": "grad", "candidates": 5_003},
        # chi2 and curvature of each candidate, as the field-scale fit reads them
        {"name": "each_100k", "kind": "each", "candidates": 100_003},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select", "select", "select", "graph", "host", "noalloc", "ingest", "align", "grad", "each"])
    if kind == "ingest":
        return {"kind": kind, "hits": _log(rng, 1, 85_000_000), "skip": rng.choice([0, 1, 2, 3]),
                "phi": rng.random() < 0.75}
    if kind in ("align", "grad", "each"):
        return {"kind": kind, "candidates": _log(rng, 1, 970_000)}
    if kind != "noalloc" and rng.random() < 0.2:
        return _select(kind, _log(rng, 1, 200_000), 15.0, 0.5, 1000, True)
    tracks = round(math.exp(rng.uniform(math.log(1.0), math.log(64.0))), 2)
    most = 262_144 if kind == "noalloc" else 1_000_000
    if tracks > 20.0:  # the work of a frame grows with the third power of its tracks
        most = int(most * (20.0 / tracks) ** 4)
    return _select(kind, _log(rng, 1, most), tracks, round(rng.uniform(0.0, 2.0), 2), rng.choice([10, 1000]))


# ------------------------------------------------------------------ inputs


def _target(n, g, dev, geo):
    u = torch.rand(2, n, generator=g, device=dev, dtype=torch.float64)
    ph = TWO_PI * torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    az = geo.target_half * (1.0 - torch.sqrt(1.0 - u[0]))
    rho = geo.target_r * (1.0 - az / geo.target_half)
    return rho * torch.cos(ph), rho * torch.sin(ph), torch.where(u[1] < 0.5, -az, az)


def _decays(n, g, dev, geo):
    """Momenta (3, n) x, y, z, of e+, e-, e+ from n decays at rest: the energies uniform over the
    three-body phase space (massless limit), an isotropic orientation."""
    u = torch.rand(2, n, generator=g, device=dev, dtype=torch.float64)
    flip = u.sum(0) < 1.0
    e1, e2 = torch.where(flip, 1.0 - u[0], u[0]), torch.where(flip, 1.0 - u[1], u[1])
    e = torch.stack([e1, e2, 2.0 - e1 - e2]) * (0.5 * geo.m_mu)
    p = torch.sqrt((e * e - geo.m_e ** 2).clamp_min(1e-6))
    c = ((p[1] ** 2 - p[0] ** 2 - p[2] ** 2) / (2.0 * p[0] * p[2])).clamp(-1.0, 1.0)
    s = torch.sqrt(1.0 - c * c)
    q = torch.randn(4, n, generator=g, device=dev, dtype=torch.float64)
    w, x, y, z = q / q.norm(dim=0)
    ax = torch.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)])   # image of the z axis
    bx = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)])   # image of the x axis
    v1, v3 = ax * p[0], bx * (p[2] * s) + ax * (p[2] * c)
    return torch.stack([v1, -(v1 + v3), v3])


def _chunk(case, phase, nf, g, dev, geo):
    """Hits of nf frames: addresses in frame order, hits per frame and, per track, the positions of its
    hits among them on the four layers (-1 where it has none).  phase: of the frames with a signal decay."""
    rate = torch.full((nf,), float(case["tracks"]), device=dev, dtype=torch.float64)
    noise = torch.full((nf,), float(case["noise"]), device=dev, dtype=torch.float64)
    if case["uneven"]:
        k = torch.exp(math.log(case["tracks"]) + torch.randn(nf, generator=g, device=dev, dtype=torch.float64))
        counts = k.round().clamp(max=400).long()
        noise = torch.where(torch.rand(nf, generator=g, device=dev) < 0.01, 100.0 * noise, noise)
    else:
        counts = torch.poisson(rate, generator=g).long()
    frames = torch.arange(nf, device=dev)
    tf = torch.repeat_interleave(frames, counts)
    n = tf.numel()
    rnd = torch.rand(4, n, generator=g, device=dev, dtype=torch.float64)
    x, y, z = _target(n, g, dev, geo)
    p = 15.0 + 38.0 * rnd[0]
    ct, psi, q = -0.8 + 1.6 * rnd[1], TWO_PI * rnd[2], torch.where(rnd[3] < 0.5, 1.0, -1.0).double()
    sf = frames[(frames + phase) % case["signal_every"] == 0]
    if sf.numel():
        v = torch.stack(_target(sf.numel(), g, dev, geo))
        mom = _decays(sf.numel(), g, dev, geo)  # (particle, axis, decay)
        pm = mom.norm(dim=1)
        tf = torch.cat([tf, sf.repeat(3)])
        x, y, z = (torch.cat([a, b.repeat(3)]) for a, b in zip((x, y, z), v))
        p, ct = torch.cat([p, pm.reshape(-1)]), torch.cat([ct, (mom[:, 2] / pm).clamp(-1, 1).reshape(-1)])
        psi = torch.cat([psi, torch.atan2(mom[:, 1], mom[:, 0]).reshape(-1)])
        q = torch.cat([q, torch.tensor([1.0, -1.0, 1.0], device=dev, dtype=torch.float64).repeat_interleave(sf.numel())])
    n = tf.numel()
    alive = torch.ones(n, device=dev, dtype=torch.bool)
    fr, ad, tr, la = [], [], [], []
    for L in range(4):
        st = torch.sqrt((1.0 - ct * ct).clamp_min(1e-12))
        rt = p * st / (geo.k * geo.B)
        cx, cy = x + q * rt * torch.sin(psi), y - q * rt * torch.cos(psi)
        d, r = torch.hypot(cx, cy).clamp_min(1e-12), float(geo.r[L])
        reach = alive & (d + rt >= r)
        a = (r * r - rt * rt + d * d) / (2.0 * d)
        h = torch.sqrt((r * r - a * a).clamp_min(0.0))
        ux, uy, a0 = cx / d, cy / d, torch.atan2(y - cy, x - cx)
        turns = []
        for s in (1.0, -1.0):
            qx, qy = a * ux - s * h * uy, a * uy + s * h * ux
            turns.append((torch.remainder(q * (a0 - torch.atan2(qy - cy, qx - cx)), TWO_PI), qx, qy))
        first = turns[0][0] <= turns[1][0]
        al, x, y = (torch.where(first, u, w) for u, w in zip(*turns))
        z = z + rt * al * ct / st
        psi = psi - q * al
        alive = reach & (z.abs() <= float(geo.H[L]))
        # multiple scattering in the layer: two orthogonal projected angles
        t1, t2 = torch.randn(2, n, generator=g, device=dev, dtype=torch.float64) * (gen.highland(1.0, geo.x0[L]) / p)
        dx = st * torch.cos(psi) - t1 * torch.sin(psi) - t2 * ct * torch.cos(psi)
        dy = st * torch.sin(psi) + t1 * torch.cos(psi) - t2 * ct * torch.sin(psi)
        dz = ct + t2 * st
        ct = (dz / torch.sqrt(dx * dx + dy * dy + dz * dz)).clamp(-1, 1)
        psi = torch.atan2(dy, dx)
        hit = alive.nonzero()[:, 0]
        nt, nr = int(geo.ntot[L]), int(geo.nrow[L])
        col = (torch.remainder(torch.atan2(y[hit], x[hit]), TWO_PI) / TWO_PI * nt).long().clamp(0, nt - 1)
        row = ((z[hit] + float(geo.H[L])) / geo.pitch).long().clamp(0, nr - 1)
        nf_hits = torch.poisson(noise, generator=g).long()
        nn = int(nf_hits.sum())
        fr += [tf[hit], torch.repeat_interleave(frames, nf_hits)]
        tr += [hit, torch.full((nn,), -1, device=dev)]
        col = torch.cat([col, torch.randint(nt, (nn,), generator=g, device=dev)])
        row = torch.cat([row, torch.randint(nr, (nn,), generator=g, device=dev)])
        nc = int(geo.ncol[L])
        ad.append(((L << 26) | ((col // nc) << 21) | ((col % nc) << 13) | row).int())
        la.append(torch.full((hit.numel() + nn,), L, device=dev))
    fr, ad, tr, la = (torch.cat(v) for v in (fr, ad, tr, la))
    shuffle = torch.randint(1 << 31, (fr.numel(),), generator=g, device=dev)
    order = torch.sort((fr << 31) | shuffle, stable=True).indices
    at = torch.empty_like(order)
    at[order] = torch.arange(order.numel(), device=dev)
    quad = torch.full((n, 4), -1, device=dev, dtype=torch.int64)
    real = tr >= 0
    quad[tr[real], la[real]] = at[real]
    return ad[order], torch.bincount(fr, minlength=nf), quad


def _frames(case, seed):
    """hits (int32), off (int64) on the GPU, and the hits of every track that reached all four layers."""
    dev = torch.device("cuda")
    geo = gen.Geometry(gen.load_config())
    g = torch.Generator(device=dev).manual_seed(seed)
    hits, counts, quads, base = [], [], [], 0
    for f0 in range(0, case["frames"], CHUNK):
        a, c, quad = _chunk(case, f0 + seed, min(CHUNK, case["frames"] - f0), g, dev, geo)
        hits.append(a)
        counts.append(c)
        if case.get("quads"):
            quads.append((quad[(quad >= 0).all(1)] + base).int())
        base += a.numel()
    off = torch.zeros(case["frames"] + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.cat(counts), 0, out=off[1:])
    return torch.cat(hits), off, torch.cat(quads) if quads else None


def _hits(case, seed):
    need = case["hits"] + case["skip"]
    hits, _, _ = _frames(_select("", need // 80 + 100, 20.0, 2.0, 1000), seed)
    return hits[case["skip"]:need]


def _candidates(case, seed):
    """Hits, offsets, frozen quadruplets whose nominal chi2 passes the track cut, and alignment parameters
    off nominal by the benchmark's misalignment."""
    n = case["candidates"]
    hits, off, quad = _frames({**_select("", n // 6 + 200, 10.0, 0.5, 10), "quads": True}, seed)
    nominal = torch.zeros(25, dtype=torch.float64, device=hits.device)
    nominal[24] = 1.0
    chi2 = torch.cat([_fit64(hits, q, nominal)[0] for q in quad.split(1 << 19)])
    cand = quad[chi2 < gen.load_config()["cuts"]["chi2_track_max"]][:n].contiguous()
    r = np.random.default_rng([seed, 0xa119])
    par = np.concatenate([r.normal(0.0, 0.050, (4, 3)), r.normal(0.0, 0.5e-3, (4, 3))], 1).reshape(-1)
    par = np.append(par, 1.0 + r.normal(0.0, 1e-3))
    assert cand.shape[0] == n
    return hits, off, cand, torch.tensor(par, dtype=torch.float32, device=hits.device)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "ctx": m3e.Context()}
    if kind == "ingest":
        s.update(hits=_hits(case, seed), phi=case["phi"])
    elif kind in ("align", "grad", "each"):
        s["hits"], s["off"], s["cand"], s["params"] = _candidates(case, seed)
    else:
        s["hits"], s["off"], _ = _frames(case, seed)
        if kind in ("select", "graph"):
            s["ctx"].prepare(case["frames"])
        if kind in ("graph", "noalloc"):
            s["keep"], s["reason"] = torch.empty(2, case["frames"], dtype=torch.uint8, device="cuda")
        if kind == "graph":
            s["graph"] = s["ctx"].graph(s["hits"], s["off"], s["keep"], s["reason"])
        if kind == "host":
            s["hits"], s["off"] = s["hits"].cpu().pin_memory(), s["off"].cpu().pin_memory()
            s["keep"], s["reason"] = (torch.empty(case["frames"], dtype=torch.uint8).pin_memory() for _ in range(2))
    return s


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "select":
        return ctx.select_frames(s["hits"], s["off"])
    if kind == "graph":
        s["graph"].launch()
        return s["keep"], s["reason"]
    if kind == "host":
        return ctx.select_frames_host(s["hits"], s["off"], s["keep"], s["reason"])
    if kind == "noalloc":
        return ctx.select_frames_noalloc(s["hits"], s["off"], s["keep"], s["reason"])
    if kind == "ingest":
        return ctx.ingest(s["hits"], with_phi=s["phi"])
    if kind == "grad":
        return ctx.fit_grad(s["hits"], s["off"], s["cand"], s["params"])
    if kind == "each":
        return (ctx.fit_chi2(s["hits"], s["off"], s["cand"], s["params"]),
                ctx.fit_kappa(s["hits"], s["off"], s["cand"], s["params"]))
    params = s["params"].detach().requires_grad_()
    loss = m3e.fit_chi2_sum(params, ctx, s["hits"], s["off"], s["cand"])
    loss.backward()
    return loss.detach(), params.grad


# ------------------------------------------------------------------ what a pass cannot do without


def _frame_ops(t, noise):
    """FP32 operations of the method on a frame of t tracks: pair tests, triplet tests, track fits, energy
    tests, vertices, from the per-item counts and the measured numbers of items of the throughput mix."""
    h = 0.95 * t + noise
    trip = 0.85 * t + 0.0028 * h ** 3
    ops = 4 * 0.65 * h * h + 6 * 0.0555 * h ** 3
    if trip > 768:
        return ops
    trk = 0.75 * t + 0.0004 * h ** 3
    combos = 0.2 * trk ** 3 / 16
    return ops + 460 * trip + 7 * trk ** 3 / 16 + (27 * combos if combos <= 1024 else 0)


def work(case):
    kind = case["kind"]
    if kind == "ingest":
        return {"bytes": case["hits"] * (20 if case["phi"] else 16), "flops": 0}
    if kind in ("align", "grad", "each"):
        n = case["candidates"]
        ops = {"align": 900 + 2600, "grad": 2600, "each": 900}[kind]
        return {"bytes": 16 * n + 16 * n + (8 * n if kind == "each" else 204), "flops": ops * n}
    nf = case["frames"]
    if case["uneven"]:  # the lognormal's quantiles
        z = [math.sqrt(2.0) * float(torch.erfinv(torch.tensor(2 * (i + 0.5) / 64 - 1))) for i in range(64)]
        ts = [min(400.0, case["tracks"] * math.exp(v)) for v in z]
    else:
        ts = [case["tracks"]]
    t = sum(ts) / len(ts)
    hits = 4 * (0.97 * t + case["noise"] * (2 if case["uneven"] else 1))
    return {"bytes": nf * (4 * hits + 8 + 2), "flops": nf * sum(_frame_ops(t, case["noise"]) for t in ts) / len(ts)}


# ------------------------------------------------------------------ 64-bit values


def _positions64(hits):
    """x, y, z, phi of packed addresses in 64 bits."""
    geo = gen.load_config()["geometry"]
    a = hits.long()
    f = lambda v: torch.tensor(v, dtype=torch.float64, device=hits.device)  # noqa: E731
    L, lad, col, row = (a >> 26) & 3, (a >> 21) & 31, (a >> 13) & 255, a & 8191
    nc = f(geo["n_cols"])[L]
    phi = (lad * nc + col + 0.5) * TWO_PI / (f(geo["n_ladders"])[L] * nc)
    r = f(geo["r_mm"])[L]
    return r * torch.cos(phi), r * torch.sin(phi), (row + 0.5) * geo["pitch_mm"] - f(geo["half_len_mm"])[L], phi


def _triplet64(a, b, c, hl, kB):
    """The multiple-scattering triplet fit of hits a -> b -> c: its linear kink model around the circle
    solution (offsets from that solution's radius), signed curvature and inverse variance."""
    u, v, w = (a - b)[:, :2], (c - b)[:, :2], (c - a)[:, :2]
    cross = u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]
    d0, d1, d2 = u.norm(dim=1), v.norm(dim=1), w.norm(dim=1)
    rt = d0 * d1 * d2 / (2.0 * cross.abs())
    ph = [2.0 * torch.atan2(cross.abs(), (-w * -v).sum(1)), 2.0 * torch.atan2(cross.abs(), (-u * w).sum(1))]
    RC, th, dphi, dth = [], [], [], []
    for d, z, f in ((d0, b[:, 2] - a[:, 2], ph[0]), (d1, c[:, 2] - b[:, 2], ph[1])):
        sh, ch = torch.sin(0.5 * f), torch.cos(0.5 * f)
        zp = z / f
        R = torch.sqrt(rt * rt + zp * zp)
        dp = -R / (d * d * ch / (8.0 * sh ** 3) + zp * zp / f)
        # dtheta / dPhi of tan(theta) = d Phi / (2 z sin(Phi/2))
        g, gp = f / (2.0 * sh), (sh - 0.5 * f * ch) / (2.0 * sh * sh)
        RC.append(R)
        th.append(torch.atan2(rt, zp))
        dphi.append(dp)
        dth.append(z * d * gp * dp / (z * z + (d * g) ** 2))
    alpha, beta = 0.5 * (dphi[0] + dphi[1]), dth[1] - dth[0]
    a0, b0 = 0.5 * dphi[1] * (RC[0] - RC[1]), th[1] - th[0] + dth[1] * (RC[0] - RC[1])
    s2 = torch.sin(0.5 * (th[0] + th[1])) ** 2
    den = alpha * alpha * s2 + beta * beta
    R = RC[0] - (alpha * a0 * s2 + beta * b0) / den
    return {"alpha": alpha, "a0": a0, "beta": beta, "b0": b0, "s2": s2, "ref": RC[0], "R": R,
            "kappa": torch.sign(cross) / R, "w": (kB * R ** 3 / hl) ** 2 * den, "hl": hl}


def _fit64(hits, cand, params):
    """chi2 and weighted mean curvature of each candidate at the given alignment; NaN where the fit fails."""
    cfg = gen.load_config()
    x0 = cfg["material"]["x_over_X0"]
    kB = cfg["constants"]["k_MeV_per_T_mm"] * cfg["field"]["B_T"] * cfg["field"]["field_scale"] * params[24]
    pts = []
    for L in range(4):
        d, w = params[6 * L:6 * L + 3], params[6 * L + 3:6 * L + 6]
        (sx, sy, sz), (cx, cy, cz), o = torch.sin(w), torch.cos(w), torch.zeros_like(w[0])
        i = o + 1.0
        Rx = torch.stack([i, o, o, o, cx, -sx, o, sx, cx]).view(3, 3)
        Ry = torch.stack([cy, o, sy, o, i, o, -sy, o, cy]).view(3, 3)
        Rz = torch.stack([cz, -sz, o, sz, cz, o, o, o, i]).view(3, 3)
        pts.append(torch.stack(_positions64(hits[cand[:, L].long()])[:3], 1) @ (Rz @ Ry @ Rx).T + d)
    fits = [_triplet64(*pts[k:k + 3], gen.highland(1.0, x0[k + 1]), kB) for k in (0, 1)]
    kb = (fits[0]["kappa"] * fits[0]["w"] + fits[1]["kappa"] * fits[1]["w"]) / (fits[0]["w"] + fits[1]["w"])
    Rb = 1.0 / kb.abs()
    chi2 = 0.0
    for f in fits:
        u = Rb - f["ref"]
        chi2 = chi2 + ((f["alpha"] * u + f["a0"]) ** 2 * f["s2"] + (f["beta"] * u + f["b0"]) ** 2) * (kB * Rb / f["hl"]) ** 2
    bad = ~((fits[0]["R"] > 0) & (fits[1]["R"] > 0) & torch.isfinite(chi2))
    return chi2.masked_fill(bad, math.nan), kb.masked_fill(bad, math.nan)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ingest":
        return tuple(_positions64(_hits(case, seed)))[:4 if case["phi"] else 3] + (() if case["phi"] else (None,))
    if kind not in ("align", "grad", "each"):
        return None  # decisions: whole numbers
    hits, off, cand, params = _candidates(case, seed)
    p = params.double().requires_grad_(kind != "each")
    if kind == "each":
        return _fit64(hits, cand, p)
    total, grad = 0.0, torch.zeros_like(p)
    for q in cand.split(1 << 18):
        with torch.no_grad():
            q = q[torch.isfinite(_fit64(hits, q, p)[0])]
        s = _fit64(hits, q, p)[0].sum()
        grad += torch.autograd.grad(s, p)[0]
        total = total + s.detach()
    return (total, grad) if kind == "align" else (total.reshape(1), grad)
