"""The engines behind the rectangle kernels, on clips that those leave to them (65 and
more rectangles): tensor-core items of 1 to 70 members with each operand type, at the
default wait limit and at a limit of the context's own, smaller markers among them; the
window scan's pruning; the mixed batch's 512x512 px class.  Records equal the oracle's."""
import functools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    return pcl


@functools.lru_cache(maxsize=None)
def _workload(px, S):
    """90 clips of 65 to 120 rectangles: shifted copies of nine, and unrelated ones"""
    W, rng = 4 * px, np.random.default_rng(px)
    c = 11
    p = W // c
    base = []
    for _ in range(18):
        k = int(rng.integers(65, 121))
        i = rng.permutation(c * c)[:k]
        j = rng.integers(0, max(2, p // 3), size=(k, 4))
        x, y = (i % c) * p, (i // c) * p
        base.append(np.stack([x + j[:, 0], y + j[:, 1], x + p - j[:, 2], y + p - j[:, 3]], 1))
    clips = [np.clip(base[i % 9] + 4 * rng.integers(-S, S + 1, size=2)[[0, 1, 0, 1]], 0, W) if i < 72 else base[i % 18]
             for i in range(90)]
    return synth.from_lists([q[(q[:, 0] < q[:, 2]) & (q[:, 1] < q[:, 3])].tolist() for q in clips], W, 4, 4 * S)


@functools.lru_cache(maxsize=None)
def _segments(px, S):
    rng = np.random.default_rng(5)
    pairs = []
    for a, k in zip(rng.permutation(90), (1, 5, 6, 10, 11, 31, 32, 33, 70)):
        pairs += [(a, b) for b in np.sort(rng.permutation(90)[:k])]
    pairs = np.array(pairs, dtype=np.int64)
    pairs = pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))]
    return pairs, oracle.ClipSet(_workload(px, S)).match(pairs, oracle.MODE_COSINE, use_gates=False)


def _equal(g, o):
    for f in ("dx_dbu", "dy_dbu", "pass_"):
        np.testing.assert_array_equal(g[f], o[f], err_msg=f)
    np.testing.assert_array_equal(g["score"].astype(np.int64), o["score"])
    assert np.abs(g["sim"].astype(np.float64) - o["sim"]).max() <= 1e-5


@pytest.mark.parametrize("limit", [0, 1_000_000_000])
@pytest.mark.parametrize("engine", ["f16", "bf16", "e4m3"])
@pytest.mark.parametrize("px,S", [(64, 4), (128, 8), (128, 5), (256, 16), (256, 7)])
def test_tensor_core_items(pcl, px, S, engine, limit):
    import torch
    wl = _workload(px, S)
    pairs, o = _segments(px, S)
    eng = {"f16": pcl.ENGINE_TC_DIRECT, "bf16": pcl.ENGINE_TC_DIRECT_BF16, "e4m3": pcl.ENGINE_TC_DIRECT_FP8}[engine]
    ctx = pcl.Context(0)
    P = pcl.params(wl.window_dbu, 4, 4 * S, cos_engine=eng, flags=pcl.P_NO_GATES)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    pcl.pcl_set_wait_limit(ctx, limit)
    tp = torch.from_numpy(pairs.astype(np.int32)).cuda()
    _equal(pcl.records_to_numpy(pcl.match(ctx, P, pcl.MODE_COSINE, cs, cs, tp)), o)
    assert pcl.pcl_device_error(ctx) == 0
    if px != 256:
        return
    # the tensor cores are reached: a limit of 1 ns runs out on them
    pcl.pcl_set_wait_limit(ctx, 1)
    pcl.match(ctx, P, pcl.MODE_COSINE, cs, cs, tp)
    with pytest.raises(pcl.PclError) as e:
        pcl.pcl_device_error(ctx)
    assert e.value.status == pcl.PCL_ERR_TIMEOUT


@pytest.mark.parametrize("px,S", [(128, 8), (256, 16), (512, 32)])
def test_scan_prunes(pcl, px, S):
    """a clip against itself: more groups than pairs (they are scanned), a quarter
    of the window at most"""
    import torch
    wl = _workload(px, S)
    ctx = pcl.Context(0)
    P = pcl.params(wl.window_dbu, 4, 4 * S, flags=pcl.P_NO_GATES,
                   cos_engine=pcl.ENGINE_FFT_PCM if px == 512 else pcl.ENGINE_EXACT_SCAN)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    groups = (2 * S + 1) * (S // 8 + (S + 7) // 8 + 1)
    pairs = np.array([[i, i] for i in range(8)])
    pcl.pcl_stats_get(ctx, reset=True)
    g = pcl.records_to_numpy(pcl.match(ctx, P, pcl.MODE_COSINE, cs, cs, torch.from_numpy(pairs.astype(np.int32)).cuda()))
    done, window = pcl.pcl_stats_get(ctx)
    assert window == len(pairs) * groups
    assert len(pairs) < done <= 0.25 * window
    _equal(g, oracle.ClipSet(wl).match(pairs, oracle.MODE_COSINE, use_gates=False))


def test_mixed_512_class_matches_oracle(pcl):
    import torch
    wl = _workload(512, 32)
    ctx = pcl.Context(0)
    P = pcl.params(2048, 4, 128, flags=pcl.P_NO_GATES)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    pairs = np.random.default_rng(1).integers(0, 90, size=(12, 2))
    pairs[:3, 1] = pairs[:3, 0] % 9 + 9
    work = np.zeros(len(pairs), pcl.WORK_DTYPE)
    work["a"], work["b"], work["mode"] = pairs[:, 0], pairs[:, 1], pcl.MODE_COSINE
    rec = torch.zeros((len(pairs), 40), dtype=torch.uint8, device="cuda")
    pcl.pcl_match_mixed(ctx, [P], [cs], torch.from_numpy(work.view(np.uint8).reshape(-1, 12)).cuda(), len(pairs), rec)
    _equal(pcl.records_to_numpy(rec), oracle.ClipSet(wl).match(pairs, oracle.MODE_COSINE, use_gates=False))
