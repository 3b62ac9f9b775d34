"""A served cosine library is its rasters: with its rectangles overwritten or not
passed at all, requests to the exact scan and the tensor-core engine give the
records of an intact library, and every aligned pair is counted by the scan."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", ["exact", "f16"])
@pytest.mark.parametrize("px", [128, 256])
def test_library_rectangles_are_not_read(px, engine):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    W = 4 * px
    wl = synth.generate(px, n_clips=400, n_seeds=20, n_copies=280, window_dbu=W, margin_dbu=W // 16, min_rects=3,
                        max_rects=12, edge_jitter=3)
    q = synth.from_lists([wl.clip(k).tolist() for k in range(40)], W, 4, wl.marker_dbu)
    ctx = pcl.Context(0)
    P = pcl.params(W, 4, W // 16, cos_engine=pcl.ENGINE_EXACT_SCAN if engine == "exact" else pcl.ENGINE_TC_DIRECT)
    want = None
    for how in ("intact", "overwritten", "missing"):
        lib = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
        pcl.pcl_rasterize(ctx, P, lib)
        if how == "overwritten":
            lib.rects.zero_()
            lib.rect_off.zero_()
        elif how == "missing":
            lib.rects = lib.rect_off = None
        pcl.pcl_stats_get(ctx, reset=True)
        srv = pcl.Server(ctx, P, lib, max_inflight=1, max_query_clips=64, cand_per_query=256, mem_budget=1 << 28)
        assert srv.submit(q.rect_off, q.rects, 7)
        done = []
        while not done:
            done = srv.poll()
        srv.close()
        assert done[0]["status"] == 0
        rec = np.sort(done[0]["records"], order=["a", "b"])
        aligned = int(((rec["flags"] & 512) > 0).sum())
        assert aligned >= 40
        if engine == "exact":  # a pair taken from its rectangles counts as one group of shifts
            assert pcl.pcl_stats_get(ctx)[0] > aligned
        want = rec if want is None else want
        np.testing.assert_array_equal(rec, want)
