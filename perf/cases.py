"""Performance cases of the pattern-similarity library.

Each case is one call (or one short sequence of calls) that a program built on
``paper_2512_13133_gb300`` makes: rasterise a clip set, generate candidate
pairs, match listed pairs with one of the engines, cache spectra, match with
re-extraction, run a mixed batch, serve query requests.  Clips are random
Manhattan layouts of the workloads the library is built for (rectangles of
sides 20-120 dbu on a 10-dbu grid, 20 dbu apart; one clip in twenty a seed, 70 %
copies of a seed with every edge moved by up to 8 dbu and the clip by up to the
marker half-width, the rest independent), generated on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2512_13133_gb300 as pcl

PITCH = 4  # dbu per pixel in every workload


def listed():
    return [
        # The plain method on a small set: 1,000 clips of 128x128 px, 3-12 rectangles, cosine 0.95 and edge
        # tolerance 4 dbu: rasters, both screens, records and the edge mode's clusters.  The smallest whole
        # run a user makes: launches, synchronisations and latency count.
        dict(name="flow_small", kind="flow", px=128, clips=1000, rmin=3, rmax=12),
        # Rasters and signatures of the 100,000-clip set (256x256 px, 5-40 rectangles), the first stage of every run.
        dict(name="raster_100k", kind="raster", px=256, clips=100_000, rmin=5, rmax=40),
        # Cosine candidates of that set (area band join, density and profile gates).
        dict(name="candidates_cosine_100k", kind="candidates", mode="cosine", px=256, clips=100_000, queries=0,
             rmin=5, rmax=40, topo=False),
        # Edge-displacement candidates of that set: the largest call of the method, 5e9 pairs.
        dict(name="candidates_edge_100k", kind="candidates", mode="edge", px=256, clips=100_000, queries=0,
             rmin=5, rmax=40, topo=False),
        # Min-Max records of a screened edge candidate list.
        dict(name="match_edge_1m", kind="match", engine="edge", px=256, pairs=1_000_000, rmin=5, rmax=40),
        # Forward transforms that the phase-correlation engine caches, for a batch of new clips.
        dict(name="spectra_4k", kind="spectra", px=256, clips=4096, rmin=5, rmax=40),
        # Phase correlation and cosine records of same-seed pairs, spectra cached (the default engine).
        dict(name="match_fft_40k", kind="match", engine="fft", px=256, pairs=40_000, rmin=5, rmax=40),
        # The same kind of list through the FP16 tensor-core correlation.
        dict(name="match_tc_fp16_100k", kind="match", engine="tc_fp16", px=256, pairs=100_000, rmin=5, rmax=40),
        # 512x512 px pairs: the exact window scan, the only cosine engine of that size.
        dict(name="match_exact512_12k", kind="match", engine="exact", px=512, pairs=12_001, rmin=5, rmax=40),
        # Re-extraction: halo rasters of a clip set, then records of its same-seed pairs.
        dict(name="halo_60k", kind="halo", px=256, pairs=60_000, rmin=5, rmax=40),
        # Mixed batch: four raster sizes, uneven (Zipf) candidate lists, half cosine and half edge items.
        dict(name="mixed_4x5k", kind="mixed", clips=5000, zipf=1.1, max_list=5000, rmin=5, rmax=40),
        # Serving: 24 requests of 1-4,096 new clips against a resident 32,768-clip library, cosine mode.
        dict(name="serve_cosine_32k", kind="serve", mode="cosine", engine="fft", px=256, clips=32_768, requests=24,
             max_query=4096, rmin=5, rmax=40),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["flow", "raster", "candidates", "candidates", "candidates", "match", "match", "match",
                       "match", "spectra", "halo", "mixed", "serve"])
    rmin, rmax = rng.choice([(3, 12), (5, 40), (5, 40)])
    base = dict(kind=kind, rmin=rmin, rmax=rmax)
    if kind == "flow":
        return dict(base, px=rng.choice([64, 128, 128, 256]), clips=_log_int(rng, 200, 4000))
    if kind == "raster":
        px = rng.choice([64, 128, 256, 256, 512])
        return dict(base, px=px, clips=_log_int(rng, 64, 100_000 if px < 512 else 20_000))
    if kind == "candidates":
        mode = rng.choice(["cosine", "edge"])
        px = rng.choice([64, 128, 256, 256, 512])
        # small rasters and few rectangles leave more pairs to the later gates
        most = 100_000 if px == 256 and rmax == 40 else 25_000
        queries = rng.choice([0, 0, 1])
        if queries:
            queries = _log_int(rng, 16, 4096)
        return dict(base, mode=mode, px=px, clips=_log_int(rng, 300, most), queries=queries,
                    topo=not queries and rng.random() < 0.15)
    if kind == "match":
        engine = rng.choice(["edge", "fft", "fft", "tc_fp16", "tc_bf16", "tc_fp8", "exact", "exact", "xysep"])
        px = rng.choice({"exact": [128, 256, 512], "edge": [64, 128, 256, 512],
                         "xysep": [64, 128, 256, 512]}.get(engine, [64, 128, 256, 256]))
        most = {"edge": 1_000_000, "xysep": 200_000, "fft": 40_000, "exact": 12_000 if px == 512 else 60_000}
        return dict(base, engine=engine, px=px, pairs=_log_int(rng, 64, most.get(engine, 100_000)))
    if kind == "spectra":
        return dict(base, px=rng.choice([64, 128, 256, 256]), clips=_log_int(rng, 16, 4096))
    if kind == "halo":
        px = rng.choice([64, 128, 256, 256, 512])
        return dict(base, px=px, pairs=_log_int(rng, 64, 60_000 if px < 512 else 6000))
    if kind == "mixed":
        return dict(base, rmin=5, rmax=40, clips=_log_int(rng, 100, 5000), zipf=1.1, max_list=_log_int(rng, 100, 5000))
    mode = rng.choice(["cosine", "cosine", "edge"])
    px = rng.choice([128, 256, 256, 512])
    engine = "exact" if px == 512 else rng.choice(["fft", "tc_fp16", "exact"])
    return dict(base, rmin=5, rmax=40, mode=mode, engine=engine, px=px, clips=_log_int(rng, 2000, 20_000),
                requests=rng.randint(1, 16), max_query=_log_int(rng, 16, 1024))


# ---------------------------------------------------------------- clips

def _marker(px):
    return px * PITCH // 16  # S = N / 16 pixels


def _uniform(gen, lo, hi, shape):
    return torch.randint(lo, hi + 1, shape, generator=gen, device="cuda", dtype=torch.int32)


def _layouts(gen, n, window, margin, rmin, rmax):
    """n random layouts on [-margin, window + margin)^2: rects [n, rmax, 4] and counts [n]"""
    rects = torch.full((n, rmax, 4), 1 << 28, dtype=torch.int32, device="cuda")  # empty places: far away
    count = torch.zeros(n, dtype=torch.int64, device="cuda")
    target = _uniform(gen, rmin, rmax, (n,)).long()
    lo = -(margin // 10)
    row = torch.arange(n, device="cuda")
    for _ in range(2 * rmax + 16):
        side = 10 * _uniform(gen, 2, 12, (n, 2))
        room = (window + margin - side) // 10 - lo + 1
        at = 10 * (lo + (torch.rand(n, 2, generator=gen, device="cuda") * room).int().clamp_(min=0))
        new = torch.cat([at, at + side], 1)
        q = rects
        apart = ((new[:, None, 2] + 20 <= q[:, :, 0]) | (q[:, :, 2] + 20 <= new[:, None, 0]) |
                 (new[:, None, 3] + 20 <= q[:, :, 1]) | (q[:, :, 3] + 20 <= new[:, None, 1]))
        ok = apart.all(1) & (count < target)
        slot = torch.where(ok, count, rmax - 1)
        rects[row, slot] = torch.where(ok[:, None], new, rects[row, slot])
        count += ok
    return rects, count


def _pack(rects, keep):
    """rectangle offsets (int32 [n + 1]) and the kept rectangles, clip after clip"""
    off = torch.zeros(keep.shape[0] + 1, dtype=torch.int32, device="cuda")
    off[1:] = keep.sum(1).cumsum(0)
    flat = rects[keep].contiguous()
    if flat.shape[0] == 0:
        flat = torch.zeros((1, 4), dtype=torch.int32, device="cuda")
    return off, flat


def _cut(rects, count, lo, hi):
    cut = rects.clamp(lo, hi)
    live = torch.arange(rects.shape[1], device="cuda")[None] < count[:, None]
    return cut, live & (cut[..., 0] < cut[..., 2]) & (cut[..., 1] < cut[..., 3])


def _clips(seed, n, px, rmin, rmax, halo=False):
    """A clip set of the workloads' recipe: (offsets, rects, labels)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 2_654_435_761 % (1 << 62) + px)
    window, margin = px * PITCH, _marker(px)
    n_seeds = max(1, n // 20)
    n_copies = int(0.7 * n)
    n_own = n - n_copies
    rects, count = _layouts(gen, n_own, window, margin, rmin, rmax)
    src = torch.randint(0, n_seeds, (n_copies,), generator=gen, device="cuda")
    copies = rects[src] + _uniform(gen, -8, 8, (n_copies, rmax, 4))
    copies[..., 2:] = torch.maximum(copies[..., 2:], copies[..., :2] + 1)
    copies += _uniform(gen, -margin, margin, (n_copies, 1, 2)).repeat(1, 1, 2)
    rects, count = torch.cat([rects, copies]), torch.cat([count, count[src]])
    label = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    label[:n_seeds] = torch.arange(n_seeds, device="cuda")
    label[n_own:] = src
    order = torch.randperm(n, generator=gen, device="cuda")
    rects, count, label = rects[order], count[order], label[order]
    h = margin if halo else 0
    off, flat = _pack(*_cut(rects, count, -h, window + h))
    return off, flat, label


def _same_seed_pairs(seed, label, m):
    """m pairs (a < b) of clips of one seed, sorted by a, then b"""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 77)
    order = torch.argsort(label, stable=True)
    sl = label[order]
    out = []
    for d in range(1, 64):  # groups hold about 15 clips
        same = (sl[d:] == sl[:-d]) & (sl[d:] >= 0)
        if not bool(same.any()):
            break
        a, b = order[:-d][same], order[d:][same]
        out.append(torch.stack([torch.minimum(a, b), torch.maximum(a, b)], 1))
    every = torch.cat(out) if out else torch.zeros((1, 2), dtype=torch.int64, device="cuda")
    pick = torch.randperm(every.shape[0], generator=gen, device="cuda")
    every = every[pick[torch.arange(m, device="cuda") % every.shape[0]]]
    every = every[torch.argsort(every[:, 0] * (1 << 32) + every[:, 1])]
    return every.int().contiguous()


ENGINES = dict(fft=pcl.ENGINE_FFT_PCM, tc_fp16=pcl.ENGINE_TC_DIRECT, tc_bf16=pcl.ENGINE_TC_DIRECT_BF16,
               tc_fp8=pcl.ENGINE_TC_DIRECT_FP8, exact=pcl.ENGINE_EXACT_SCAN, xysep=pcl.ENGINE_XYSEP)


def _params(px, engine="fft", flags=0):
    if engine == "exact" and px == 512:
        engine = "fft"  # 512x512 px takes the exact scan by itself
    return pcl.params(px * PITCH, PITCH, _marker(px), cos_engine=ENGINES.get(engine, 0), flags=flags)


def _rasterised(ctx, P, off, rects, with_spec=False):
    cs = pcl.alloc_clipset(P, off, rects.reshape(-1), with_spec=with_spec)
    pcl.pcl_rasterize(ctx, P, cs)
    return cs


def _match_clips(case):
    return case["pairs"] // 5 + 200  # about 5.6 same-seed pairs per clip


# ---------------------------------------------------------------- prepare

def prepare(case, seed):
    s = {"case": case, "ctx": pcl.Context(0)}
    ctx, kind = s["ctx"], case["kind"]
    if kind == "mixed":
        return _prepare_mixed(s, case, seed)
    px, shape = case["px"], (case["rmin"], case["rmax"])
    if kind in ("flow", "raster"):
        off, rects, _ = _clips(seed, case["clips"], px, *shape)
        s["P"] = _params(px)
        room = torch.zeros((case["clips"] * case["rmax"], 4), dtype=torch.int32, device="cuda")
        room[:rects.shape[0]] = rects
        s["cs"] = pcl.alloc_clipset(s["P"], off, room.reshape(-1), with_spec=kind == "flow")
        s["cs"].rorder.zero_()
    elif kind == "candidates":
        s["P"] = _params(px, flags=pcl.P_TOPO_HASH if case["topo"] else 0)
        s["mode"] = pcl.MODE_COSINE if case["mode"] == "cosine" else pcl.MODE_EDGE
        n, q = case["clips"], case["queries"]
        off, rects, _ = _clips(seed, n + q, px, *shape)
        cs = _rasterised(ctx, s["P"], off, rects)
        s["cs"], s["b"] = (cs.view(s["P"], 0, q), cs.view(s["P"], q, n + q)) if q else (cs, None)
        s["all"] = cs
        s["cap"] = 1 << 22 if case["mode"] == "edge" else 1 << 16
    elif kind == "match":
        s["P"] = _params(px, case["engine"], 0 if case["engine"] == "edge" else pcl.P_NO_GATES)
        s["mode"] = pcl.MODE_EDGE if case["engine"] == "edge" else pcl.MODE_COSINE
        m = case["pairs"]
        if case["engine"] == "edge":  # the screen's survivors, about one pair in 2,000
            n = int(min(100_000, 64 + math.sqrt(m * 4400)))
            off, rects, label = _clips(seed, n, px, *shape)
            s["cs"] = _rasterised(ctx, s["P"], off, rects)
            pairs, _ = pcl.candidates(ctx, s["P"], s["mode"], s["cs"], cap=1 << 22)
            if pairs.shape[0]:
                keys = torch.sort(pairs[:, 0].long() * (1 << 32) + pairs[:, 1]).values
                keys = keys[torch.arange(m, device="cuda") * keys.shape[0] // m]
                s["pairs"] = torch.stack([keys >> 32, keys & 0xFFFFFFFF], 1).int().contiguous()
            else:
                s["pairs"] = _same_seed_pairs(seed, label, m)
        else:
            off, rects, label = _clips(seed, _match_clips(case), px, *shape)
            spectra = case["engine"] == "fft"
            s["cs"] = _rasterised(ctx, s["P"], off, rects, with_spec=spectra)
            if spectra:
                pcl.pcl_spectra(ctx, s["P"], s["cs"])
            s["pairs"] = _same_seed_pairs(seed, label, m)
    elif kind == "spectra":
        off, rects, _ = _clips(seed, case["clips"], px, *shape)
        s["P"] = _params(px)
        s["cs"] = _rasterised(ctx, s["P"], off, rects, with_spec=True)
        s["list"] = torch.arange(case["clips"], dtype=torch.int32, device="cuda")
    elif kind == "halo":
        off, rects, label = _clips(seed, _match_clips(case), px, *shape, halo=True)
        s["P"] = _params(px)
        s["cs"] = _rasterised(ctx, s["P"], off, rects)
        s["hbits"], s["norms"] = pcl.alloc_halo(s["P"], s["cs"])
        s["pairs"] = _same_seed_pairs(seed, label, case["pairs"])
        s["rec"] = torch.zeros((case["pairs"], 40), dtype=torch.uint8, device="cuda")
    elif kind == "serve":
        _prepare_serve(s, case, seed)
    return s


def _prepare_mixed(s, case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 13)
    n, most = case["clips"], case["max_list"]
    cdf = torch.arange(1, most + 1, dtype=torch.float64, device="cuda").pow(-case["zipf"]).cumsum(0)
    s["params"], s["sets"], work = [], [], []
    for k, px in enumerate((64, 128, 256, 512)):
        P = _params(px)
        off, rects, label = _clips(seed * 4 + k, n, px, case["rmin"], case["rmax"])
        s["params"].append(P)
        s["sets"].append(_rasterised(s["ctx"], P, off, rects, with_spec=px <= 256))
        # Zipf list lengths; half of the partners from the clip's own seed group
        u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]
        length = (torch.searchsorted(cdf, u) + 1).clamp_(max=most)
        a = torch.repeat_interleave(torch.arange(n, device="cuda"), length)
        b = torch.randint(0, n, a.shape, generator=gen, device="cuda")
        order = torch.argsort(label, stable=True)
        first = torch.searchsorted(label[order], label)
        size = torch.searchsorted(label[order], label, right=True) - first
        same = (torch.rand(a.shape, generator=gen, device="cuda") < 0.5) & (label[a] >= 0) & (size[a] > 1)
        mate = order[first[a] + (torch.rand(a.shape, generator=gen, device="cuda") * size[a]).long().clamp_(max=n - 1)
                     .minimum(size[a] - 1)]
        b = torch.where(same, mate, b)
        a, b = a[a != b], b[a != b]
        # a fixed number of items, in list order
        m = int(0.9 * n * float(torch.arange(1, most + 1, device="cuda", dtype=torch.float64).pow(1 - case["zipf"]).sum()
                                / cdf[-1])) + 1
        pick = torch.randperm(a.shape[0], generator=gen, device="cuda")
        pick = pick[torch.arange(m, device="cuda") % a.shape[0]].sort().values
        a, b = a[pick], b[pick]
        mode = 1 + (torch.rand(a.shape, generator=gen, device="cuda") < 0.5).long()
        work.append(torch.stack([a, b, k + (mode << 16)], 1))
    work = torch.cat(work).int()
    cosine = (work[:, 2] >> 16) == 1
    s["work"] = torch.cat([work[cosine], work[~cosine]]).contiguous().view(torch.uint8)
    s["n_cosine"] = int(cosine.sum())
    s["rec"] = torch.zeros((work.shape[0], 40), dtype=torch.uint8, device="cuda")
    s["tune"] = pcl.Tuning(2, 0, 64)
    return s


def _prepare_serve(s, case, seed):
    px, n = case["px"], case["clips"]
    window = px * PITCH
    engine = case["engine"]
    s["P"] = _params(px, engine)
    mode = pcl.MODE_COSINE if case["mode"] == "cosine" else pcl.MODE_EDGE
    off, rects, _ = _clips(seed, n, px, case["rmin"], case["rmax"])
    s["cs"] = _rasterised(s["ctx"], s["P"], off, rects,
                          with_spec=mode == pcl.MODE_COSINE and engine == "fft" and px <= 256)
    s["server"] = pcl.Server(s["ctx"], s["P"], s["cs"], max_inflight=8, max_query_clips=case["max_query"],
                             max_query_rects=case["max_query"] * 48, mode=mode, mem_budget=12 << 30,
                             cand_per_query=128 if mode == pcl.MODE_COSINE else 4096, pass_copy=1 << 16)
    # query clips: library clips moved by up to 8 dbu and cut to the window
    r = np.random.default_rng(seed)
    sizes = np.random.default_rng(case["requests"])  # the request sizes are the case's
    offs, flat = off.cpu().numpy().astype(np.int64), rects.cpu().numpy()
    s["requests"] = []
    for _ in range(case["requests"]):
        k = int(min(case["max_query"], max(1, round(math.exp(sizes.uniform(0, math.log(case["max_query"])))))))
        pick = r.integers(0, n, size=k)
        lens = offs[pick + 1] - offs[pick]
        clip = np.repeat(np.arange(k), lens)
        at = np.repeat(offs[pick], lens) + np.arange(lens.sum()) - np.repeat(np.cumsum(lens) - lens, lens)
        move = r.integers(-8, 9, size=(k, 2))
        q = np.clip(flat[at] + np.concatenate([move, move], 1)[clip], 0, window)
        live = (q[:, 0] < q[:, 2]) & (q[:, 1] < q[:, 3])
        ro = np.zeros(k + 1, np.uint32)
        ro[1:] = np.cumsum(np.bincount(clip[live], minlength=k))
        s["requests"].append((ro, np.ascontiguousarray(q[live], np.int32)))
    queries = sum(ro.shape[0] - 1 for ro, _ in s["requests"])
    s["rows"] = queries * (4 if mode == pcl.MODE_COSINE else 64) + 64


# ---------------------------------------------------------------- run

def run(s):
    return globals()["_run_" + s["case"]["kind"]](s)


def _records(rec):
    """the similarity and the whole-number fields of a record list"""
    w = rec.view(torch.int32)
    return {"sim": w[:, 4].view(torch.float32), "place": w[:, :4], "fields": w[:, 5:]}


def _sorted_pairs(pairs):
    return torch.sort(pairs.view(torch.int64).view(-1)).values.view(torch.int32).view(-1, 2)


def _table(rows, cap):
    """rows in a table of cap rows, zeros after them"""
    return torch.nn.functional.pad(rows[:cap], (0, 0, 0, max(0, cap - rows.shape[0])))


def _sets(cs):
    n, N = cs.n, cs.N
    nb = N // 16
    size = dict(bits=n * N * N // 8, pop=4 * n, prof=4 * n * N, blk=4 * n * nb * nb, esig=32 * n, occ=512 * n,
                rorder=int(cs.rects.numel()) // 2)
    wide = dict(bits=torch.int64, occ=torch.int64, pop=torch.int32, esig=torch.int32, prof=torch.int16,
                blk=torch.int16, rorder=torch.int16)
    return {k: getattr(cs, k)[:v].view(wide[k]) for k, v in size.items()}


def _run_flow(s):
    ctx, P, cs = s["ctx"], s["P"], s["cs"]
    pcl.pcl_rasterize(ctx, P, cs)
    out = {}
    for name, mode in (("cosine", pcl.MODE_COSINE), ("edge", pcl.MODE_EDGE)):
        pairs, gates = pcl.candidates(ctx, P, mode, cs)
        pairs = _sorted_pairs(pairs)
        rec = pcl.match(ctx, P, mode, cs, cs, pairs)
        out[name] = {"gates": gates, "rec": _table(rec.view(torch.int32), 1 << 15)}
    r = pcl.records_to_numpy(rec)
    relaxed = ((r["flags"] & pcl.F_EDGE_VERIFY_FAIL) == 0) & (r["score"] <= P.edge_tol_dbu + 2)
    rep, clusters, rounds = pcl.pcl_cluster_loop(np.stack([r["a"], r["b"]], 1), r["pass_"], relaxed, cs.n)
    out["rep"], out["clusters"] = rep, clusters
    return out


def _run_raster(s):
    pcl.pcl_rasterize(s["ctx"], s["P"], s["cs"])
    return _sets(s["cs"])


def _run_candidates(s):
    pairs, gates = pcl.candidates(s["ctx"], s["P"], s["mode"], s["cs"], cap=s["cap"], b=s["b"])
    return {"pairs": _table(_sorted_pairs(pairs), s["cap"]), "gates": gates}


def _run_match(s):
    return _records(pcl.match(s["ctx"], s["P"], s["mode"], s["cs"], s["cs"], s["pairs"]))


def _run_spectra(s):
    cs = s["cs"]
    pcl.pcl_spectra(s["ctx"], s["P"], cs, s["list"])
    return cs.spec[:cs.n * cs.L * cs.Ls * 8].view(torch.float32).view(cs.n, cs.L, cs.Ls, 2)[:, :, :cs.L // 2 + 1]


def _run_halo(s):
    pcl.pcl_rasterize_halo(s["ctx"], s["P"], s["cs"], s["hbits"], s["norms"])
    pcl.pcl_match_halo(s["ctx"], s["P"], s["cs"], s["cs"], s["hbits"], s["norms"], s["pairs"], s["rec"])
    return _records(s["rec"])


def _run_mixed(s):
    pcl.pcl_match_mixed(s["ctx"], s["params"], s["sets"], s["work"], s["n_cosine"], s["rec"], s["tune"])
    return s["rec"].view(torch.int32)


def _run_serve(s):
    srv, todo = s["server"], s["requests"]
    done, sent = [None] * len(todo), 0
    left = len(todo)
    while left:
        if sent < len(todo) and srv.submit(*todo[sent], sent):
            sent += 1
            continue
        for c in srv.poll():
            done[c["id"]] = c
            left -= 1
    count = np.array([(c["status"], c["n_candidates"], c["pass_pairs"].shape[0]) for c in done])
    rec = np.concatenate([c["records"] for c in done])
    # by request, then library clip and query clip
    req = np.repeat(np.arange(len(done), dtype=np.uint64), [c["records"].shape[0] for c in done])
    key = (req << np.uint64(32)) | (rec["a"].astype(np.uint64) << np.uint64(17)) | rec["b"].astype(np.uint64)
    out = np.zeros((s["rows"], 10), np.int32)
    rec = rec[np.argsort(key)].view(np.int32).reshape(-1, 10)[:s["rows"]]
    out[:rec.shape[0]] = rec
    return {"count": count, "rec": out}


# ---------------------------------------------------------------- work

def _set_bytes(px):
    """raster and signatures of one clip"""
    nb = px // 16
    return px * px // 8 + 4 + 4 * px + 4 * nb * nb + 32 + 512


def work(case):
    kind = case["kind"]
    rect = 18 * (case["rmin"] + case["rmax"]) / 2  # rectangles and their order, one clip
    if kind == "mixed":
        items = 4 * case["clips"] * min(360.0, case["max_list"] / 8)
        return {"bytes": case["clips"] * sum(_set_bytes(p) + rect for p in (64, 128, 256, 512)) + 52 * items,
                "flops": 0}
    px = case["px"]
    L, side = 9 * px // 8, 2 * (px // 16) + 1
    spec = 8 * L * (L // 2 + 1)
    if kind in ("flow", "raster"):
        return {"bytes": case["clips"] * (_set_bytes(px) + rect), "flops": 0}
    if kind == "candidates":
        n = case["clips"] + case["queries"]
        one = 4 + 4 * px + 4 * (px // 16) ** 2 if case["mode"] == "cosine" else 32 + 512 + rect
        return {"bytes": n * one, "flops": 0}
    if kind == "spectra":
        return {"bytes": case["clips"] * (px * px // 8 + spec), "flops": case["clips"] * 2.5 * L * L * math.log2(L * L)}
    if kind == "serve":
        q = case["requests"] * case["max_query"] / max(1.0, math.log(case["max_query"]))
        return {"bytes": (case["clips"] + q) * _set_bytes(px), "flops": 0}
    m = case["pairs"]
    if kind == "halo":
        return {"bytes": _match_clips(case) * (px * px // 8 + 2 * (px + px // 8) ** 2 // 8) + 48 * m, "flops": 0}
    engine = case["engine"]
    if engine in ("edge", "xysep"):
        return {"bytes": 48 * m + math.sqrt(m * 4400) * (544 + rect), "flops": 0}
    one = spec + px * px // 8 if engine == "fft" else px * px // 8
    flops = 2.0 * side * side * px * px * m if engine.startswith("tc") else 0
    return {"bytes": _match_clips(case) * one + 48 * m, "flops": flops}


# ---------------------------------------------------------------- exact

def _images(off, rects, ids, px, halo=0):
    """0/1 rasters (float64 [k, px + 2 halo, px + 2 halo]) of the listed clips: pixel centres in some rectangle"""
    at = (torch.arange(-halo, px + halo, device="cuda") * PITCH + PITCH // 2)[None, None]
    off = off.long()
    lens = (off[1:] - off[:-1])[ids]
    k = torch.arange(int(lens.max().clamp(min=1)), device="cuda")
    q = rects[(off[ids][:, None] + k).clamp(max=rects.shape[0] - 1)]
    live = (k[None] < lens[:, None])[..., None]
    x = ((q[..., 0:1] <= at) & (at < q[..., 2:3]) & live).float()
    y = ((q[..., 1:2] <= at) & (at < q[..., 3:4])).float()
    return (torch.einsum("kry,krx->kyx", y, x) > 0).double()


def _exact_sims(off, rects, pairs, px, halo):
    S = px // 16
    L = px + 2 * S
    out = []
    step = max(8, 2_000_000 // (px * px) * 8)
    ones = torch.fft.rfft2(torch.ones((px, px), dtype=torch.float64, device="cuda"), s=(L, L)).conj()
    for p in pairs.long().split(step):
        A = _images(off, rects, p[:, 0], px)
        B = _images(off, rects, p[:, 1], px, S if halo else 0)
        FB = torch.fft.rfft2(B, s=(L, L))
        c = torch.fft.irfft2(torch.fft.rfft2(A, s=(L, L)).conj() * FB, s=(L, L)).round()
        pa = A.sum((1, 2))[:, None, None]
        if halo:  # B(x + t), t in [0, 2S]: the moved window of the member
            c = c[:, :2 * S + 1, :2 * S + 1]
            n = torch.fft.irfft2(ones * FB, s=(L, L)).round()[:, :2 * S + 1, :2 * S + 1]
        else:  # shifts |t| <= S of the circular correlation
            t = torch.arange(-S, S + 1, device="cuda") % L
            c = c[:, t][:, :, t]
            n = B.sum((1, 2))[:, None, None].expand_as(c)
        sim = torch.where((pa > 0) & (n > 0), c / (pa * n).clamp(min=1).sqrt(), ((pa == 0) & (n == 0)).double())
        out.append(sim.amax((1, 2)))
    return torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectra":
        px = case["px"]
        off, rects, _ = _clips(seed, case["clips"], px, case["rmin"], case["rmax"])
        L = 9 * px // 8
        ids = torch.arange(case["clips"], device="cuda")
        return torch.cat([torch.view_as_real(torch.fft.rfft2(_images(off, rects, i, px), s=(L, L)))
                          for i in ids.split(256)])
    if kind == "halo" or (kind == "match" and case["engine"] not in ("edge", "xysep")):
        halo = kind == "halo"
        off, rects, label = _clips(seed, _match_clips(case), case["px"], case["rmin"], case["rmax"], halo=halo)
        pairs = _same_seed_pairs(seed, label, case["pairs"])
        return {"sim": _exact_sims(off, rects, pairs, case["px"], halo), "place": None, "fields": None}
    return None
