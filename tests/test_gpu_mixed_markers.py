"""A mixed batch with a 512x512 px class whose marker is past N/16, up to the widest
one: its cosine items are reported as unsupported, and its edge items and the
other class's items get the records of their own entry points."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("items", ["all", "edge of the large class"])
@pytest.mark.parametrize("S", [32, 33, 59, 60, 64])
def test_wide_markers_at_512(S, items):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    ctx = pcl.Context(0)
    Ps, sets, work = [], [], []
    rng = np.random.default_rng(S)
    for c, (px, s) in enumerate([(64, 4), (512, S)]):
        wl = synth.generate(px, n_clips=24, n_seeds=4, n_copies=16, window_dbu=4 * px, margin_dbu=px // 4, min_rects=2,
                            max_rects=max(4, px // 16), edge_jitter=3)
        P = pcl.params(4 * px, 4, 4 * s)
        cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=px < 512)
        pcl.pcl_rasterize(ctx, P, cs)
        Ps.append(P)
        sets.append(cs)
        for mode in (pcl.MODE_COSINE, pcl.MODE_EDGE):
            if items != "all" and mode == pcl.MODE_COSINE and c == 1:
                continue
            w = np.zeros(120, pcl.WORK_DTYPE)
            w["a"], w["b"] = rng.integers(0, wl.n, size=(2, len(w)))
            w["a"][:30] = w["b"][:30]
            w["cls"], w["mode"] = c, mode
            work.append(w)
    work = np.concatenate(work)
    work = work[np.argsort(work["mode"], kind="stable")]
    n_cos = int((work["mode"] == pcl.MODE_COSINE).sum())
    rec = torch.zeros((len(work), 40), dtype=torch.uint8, device="cuda")
    pcl.pcl_match_mixed(ctx, Ps, sets, torch.from_numpy(work.view(np.uint8).reshape(-1, 12)).cuda(), n_cos, rec)
    g = pcl.records_to_numpy(rec)
    for c in (0, 1):
        for mode in (pcl.MODE_COSINE, pcl.MODE_EDGE):
            sel = np.flatnonzero((work["cls"] == c) & (work["mode"] == mode))
            if len(sel) == 0:
                continue
            if mode == pcl.MODE_COSINE and c == 1 and S > 32:
                assert (g["flags"][sel] == pcl.GATE_UNSUPPORTED).all()
                continue
            pairs = np.stack([work["a"][sel], work["b"][sel]], 1).astype(np.int32)
            r = pcl.records_to_numpy(pcl.match(ctx, Ps[c], mode, sets[c], sets[c], torch.from_numpy(pairs).cuda()))
            for f in ("a", "b", "dx_dbu", "dy_dbu", "score", "pass_", "mode"):
                np.testing.assert_array_equal(g[f][sel], r[f], err_msg=f"class {c} mode {mode} field {f}")
            assert ((r["flags"] & pcl.F_ALIGNED) > 0).any()
