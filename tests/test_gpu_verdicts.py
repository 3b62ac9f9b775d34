"""Long lists over few clips, where each clip is compared with its raster once before
the pairs: rectangles written again after the rasters were made, one set and two, lists
cut short on the device above and below the rule's line, indices out of range and empty
sets.  Records equal the oracle's, and none past the count is written."""
import functools

import numpy as np
import pytest

import oracle
from test_gpu_halo_source import _rewritten as _rewritten_halo
from test_gpu_halo_source import _workload as _workload_halo
from test_gpu_rect_source import _rewritten, _workload

pytestmark = pytest.mark.gpu
N = 4600  # the rule's line: 4,096 pairs and twice the clips


@pytest.fixture(scope="module")
def pcl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    return pcl


@functools.lru_cache(maxsize=None)
def _case(px, halo):
    wl = _workload_halo(px) if halo else _workload(px)
    rng = np.random.default_rng(px)
    some = rng.integers(0, wl.n, size=(40 if px == 512 else 150, 2))
    some[:4] = [[wl.n - 1, wl.n - 1], [wl.n - 2, wl.n - 2], [wl.n - 2, wl.n - 1], [0, 0]]
    o = oracle.ClipSet(wl, halo=True).match(some, oracle.MODE_COSINE_HALO) if halo else \
        oracle.ClipSet(wl).match(some, oracle.MODE_COSINE, use_gates=False)
    pick = np.sort(rng.integers(0, len(some), size=N))
    pick = pick[np.lexsort((some[pick, 1], some[pick, 0]))]
    return wl, some[pick], o[pick]


def _check(rec, pcl, o, count):
    assert not rec[count:].any()
    g = pcl.records_to_numpy(rec)[:count]
    for f in ("dx_dbu", "dy_dbu", "pass_"):
        np.testing.assert_array_equal(g[f], o[f][:count], err_msg=f)
    np.testing.assert_array_equal(g["score"].astype(np.int64), o["score"][:count])
    assert np.abs(g["sim"].astype(np.float64) - o["sim"][:count]).max() <= 1e-5
    return g


@pytest.mark.parametrize("sets", ["one", "members written again", "representatives written again"])
@pytest.mark.parametrize("how", ["intact", "mirrored", "doubled"])
@pytest.mark.parametrize("px,engine", [(128, "exact"), (256, "exact"), (256, "f16"), (64, "f16"), (512, "exact")])
def test_pairs(pcl, px, engine, how, sets):
    import torch
    wl, pairs, o = _case(px, False)
    ctx = pcl.Context(0)
    e = pcl.ENGINE_TC_DIRECT if engine == "f16" else pcl.ENGINE_FFT_PCM if px == 512 else pcl.ENGINE_EXACT_SCAN
    P = pcl.params(4 * px, 4, px // 4, cos_engine=e, flags=pcl.P_NO_GATES)
    a, b = (pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False) for _ in range(2))
    if sets == "one":
        b = a
    for c in (a, b):
        pcl.pcl_rasterize(ctx, P, c)
    if how != "intact":
        (a if sets.startswith("rep") else b).rects.copy_(torch.from_numpy(_rewritten(wl, how).reshape(-1)))
    tp = torch.from_numpy(pairs.astype(np.int32)).cuda()
    for count in (N, 4200, 4095):
        rec = torch.zeros((N, 40), dtype=torch.uint8, device="cuda")
        pcl.pcl_match_pairs(ctx, P, pcl.MODE_COSINE, a, b, tp, rec,
                            d_n=torch.tensor([count], dtype=torch.int64, device="cuda") if count < N else None)
        assert not _check(rec, pcl, o, count)["reserved"].any()
    assert pcl.pcl_device_error(ctx) == 0


@pytest.mark.parametrize("side", ["representatives", "members"])
@pytest.mark.parametrize("how", ["intact", "mirrored", "doubled", "cut"])
@pytest.mark.parametrize("px", [64, 256])
def test_reextraction(pcl, px, how, side):
    import torch
    wl, pairs, o = _case(px, True)
    ctx = pcl.Context(0)
    P = pcl.params(4 * px, 4, px // 4)
    a, b = (pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False) for _ in range(2))
    pcl.pcl_rasterize(ctx, P, a)
    hb, nb = pcl.alloc_halo(P, b)
    pcl.pcl_rasterize_halo(ctx, P, b, hb, nb)
    if how != "intact":
        (a if side == "representatives" else b).rects.copy_(torch.from_numpy(_rewritten_halo(wl, how)))
    tp = torch.from_numpy(pairs.astype(np.int32)).cuda()
    for count in (N, 4200, 4095):
        rec = torch.zeros((N, 40), dtype=torch.uint8, device="cuda")
        pcl.pcl_match_halo(ctx, P, a, b, hb, nb, tp, rec,
                           d_n=torch.tensor([count], dtype=torch.int64, device="cuda") if count < N else None)
        g = _check(rec, pcl, o, count)
        np.testing.assert_array_equal(g["reserved"].astype(np.int64), o["pad"][:count].astype(np.int64))


@pytest.mark.parametrize("halo", [False, True])
@pytest.mark.parametrize("na,nb", [(0, 0), (0, 22), (22, 0), (5, 22)])
def test_indices_out_of_range(pcl, na, nb, halo):
    import torch
    wl, pairs, o = _case(64 if halo else 128, halo)
    ctx = pcl.Context(0)
    px = 64 if halo else 128
    P = pcl.params(4 * px, 4, px // 4, cos_engine=pcl.ENGINE_EXACT_SCAN, flags=pcl.P_NO_GATES)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    a, b = cs.view(P, 0, na), cs.view(P, 0, nb)
    tp = torch.from_numpy(pairs.astype(np.int32)).cuda()
    rec = torch.zeros((N, 40), dtype=torch.uint8, device="cuda")
    if halo:
        h, nrm = pcl.alloc_halo(P, cs)
        pcl.pcl_rasterize_halo(ctx, P, cs, h, nrm)
        pcl.pcl_match_halo(ctx, P, a, b, h, nrm, tp, rec)
    else:
        pcl.pcl_match_pairs(ctx, P, pcl.MODE_COSINE, a, b, tp, rec)
    g = pcl.records_to_numpy(rec)
    bad = (pairs[:, 0] >= na) | (pairs[:, 1] >= nb)
    assert (g["flags"][bad] == pcl.GATE_BAD_INDEX).all()
    np.testing.assert_array_equal(g["score"][~bad].astype(np.int64), o["score"][~bad])
