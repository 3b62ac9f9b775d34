"""A rectangle without a pixel centre shares no pixel: re-extraction pairs of clips
that hold one beside a rectangle over the window's origin are taken from their
rectangles (one group of shifts a pair), with the oracle's records."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("px", [64, 256])
def test_slivers_share_no_pixel(px):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    W, m = 4 * px, px // 4
    over = [-m // 2, -m // 2, W // 4, W // 5]
    wide, tall = [W // 2, W // 2, W - 8, W // 2 + 1], [W // 2 - 3, W // 3, W // 2 - 2, W - 40]
    clips = [[over, wide], [tall, over], [wide, tall, over, [W // 2, 9, W - 9, W // 3]], [over]]
    wl = synth.from_lists(clips, W, 4, m)
    P = pcl.params(W, 4, m)
    ctx = pcl.Context(0)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    hb, nb = pcl.alloc_halo(P, cs)
    pcl.pcl_rasterize_halo(ctx, P, cs, hb, nb)
    pairs = np.stack(np.meshgrid(np.arange(4), np.arange(4), indexing="ij"), -1).reshape(-1, 2)
    rec = torch.zeros((16, 40), dtype=torch.uint8, device="cuda")
    pcl.pcl_stats_get(ctx, reset=True)
    pcl.pcl_match_halo(ctx, P, cs, cs, hb, nb, torch.from_numpy(pairs.astype(np.int32)).cuda(), rec)
    assert pcl.pcl_stats_get(ctx, kernel="halo")[0] == 16
    g = pcl.records_to_numpy(rec)
    o = oracle.ClipSet(wl, halo=True).match(pairs.astype(np.int64), oracle.MODE_COSINE_HALO)
    for f in ("dx_dbu", "dy_dbu", "pass_"):
        np.testing.assert_array_equal(g[f], o[f], err_msg=f)
    np.testing.assert_array_equal(g["score"].astype(np.int64), o["score"])
