"""Pending cosine items of a mixed batch that lie side by side in the list (one clip's,
one class's, 512x512 px clips that the rectangle kernel leaves to the scan), in lists
from one item to several claims per CTA: records equal the classes' own entry points', and
a short list is spread over the GPU."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def batch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    ctx = pcl.Context(0)
    Ps, sets = [], []
    rng = np.random.default_rng(4)
    for px in (64, 256, 512):
        W = 4 * px
        wl = synth.generate(px, n_clips=30, n_seeds=3, n_copies=27, window_dbu=W, margin_dbu=W // 16, min_rects=3,
                            max_rects=10, edge_jitter=2)
        clips = [wl.clip(i).tolist() for i in range(wl.n)]
        if px == 512:  # rectangles sharing pixels: none of its items is decided from rectangles
            clips = [c + [[x + 4, y + 4, X, Y] for x, y, X, Y in c[:1]] for c in clips]
        wl = synth.from_lists(clips, W, 4, W // 16)
        P = pcl.params(W, 4, W // 16, cos_num=80)
        cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=px < 512)
        pcl.pcl_rasterize(ctx, P, cs)
        Ps.append(P)
        sets.append(cs)
    return pcl, ctx, Ps, sets, rng


def _run(batch, work):
    import torch
    pcl, ctx, Ps, sets, _ = batch
    rec = torch.zeros((len(work), 40), dtype=torch.uint8, device="cuda")
    tw = torch.from_numpy(work.view(np.uint8).reshape(-1, 12)).cuda()
    call = lambda: pcl.pcl_match_mixed(ctx, Ps, sets, tw, len(work), rec)
    call()
    return rec, call


@pytest.mark.parametrize("sizes", [(1, 0, 0), (0, 0, 1), (31, 33, 32), (500, 700, 90), (3, 40000, 0), (90000, 5, 33)])
def test_items_side_by_side(batch, sizes):
    import torch
    pcl, ctx, Ps, sets, rng = batch
    parts = []
    for c, k in enumerate(sizes):
        w = np.zeros(k, pcl.WORK_DTYPE)
        w["a"], w["b"] = rng.integers(0, 30, size=(2, k))
        w["b"][:k // 2] = w["a"][:k // 2]  # the first half of a class is pending throughout
        w["cls"], w["mode"] = c, pcl.MODE_COSINE
        parts.append(w)
    work = np.concatenate(parts)
    g = pcl.records_to_numpy(_run(batch, work)[0])
    for c, k in enumerate(sizes):
        if k == 0:
            continue
        sel = work["cls"] == c
        tp = torch.from_numpy(np.stack([work["a"][sel], work["b"][sel]], 1).astype(np.int32)).cuda()
        r = pcl.records_to_numpy(pcl.match(ctx, Ps[c], pcl.MODE_COSINE, sets[c], sets[c], tp))
        for f in ("a", "b", "dx_dbu", "dy_dbu", "score", "pass_", "mode", "flags"):
            np.testing.assert_array_equal(g[f][sel], r[f], err_msg=f"class {c} field {f}")


@pytest.mark.parametrize("cls", [1, 2])
def test_short_lists_use_the_whole_gpu(batch, cls):
    """2,048 pending items side by side take no longer than a few dozen times 16 of
    them (a claim of 512 consecutive ones: 4 CTAs of 152 and more)"""
    import torch
    pcl = batch[0]
    times = {}
    for n in (16, 2048):
        work = np.zeros(n, pcl.WORK_DTYPE)
        work["a"] = work["b"] = 3
        work["cls"], work["mode"] = cls, pcl.MODE_COSINE
        _, call = _run(batch, work)
        best = float("inf")
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times[n] = best
    assert times[2048] < 12 * times[16], times
