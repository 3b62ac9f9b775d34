"""The rasters are what a cosine record is about: a rectangle buffer written again
after the rasters were made (mirrored, moved by a pixel, one rectangle doubled
onto another of its size, another set's rectangles) changes no record of the
exact scan, the tensor-core engine or the mixed batch's 512x512 px class."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.fixture(scope="module")
def ctx(torch_cuda):
    import paper_2512_13133_gb300 as pcl
    return pcl.Context(0)


def _workload(px, halo=False):
    W, m = 4 * px, px // 4
    wl = synth.generate(px, n_clips=20, n_seeds=4, n_copies=12, window_dbu=W, margin_dbu=m, min_rects=2,
                        max_rects=max(4, px // 16), edge_jitter=3, halo_dbu=m if halo else 0)
    clips = [wl.clip(i).tolist() for i in range(wl.n)]
    s = W // 8  # two squares of one size: doubled, their areas still add up to the raster's ones
    clips += [[[s, s, 2 * s, 2 * s], [5 * s, 4 * s, 6 * s, 5 * s]], [[s, s, 3 * s, 2 * s], [4 * s, 5 * s, 6 * s, 6 * s]]]
    return synth.from_lists(clips, W, 4, m)


def _rewritten(wl, how):
    r = wl.rects.copy()
    if how == "mirrored":
        r[:, [0, 2]] = wl.window_dbu - wl.rects[:, [2, 0]]
    elif how == "moved":
        r += np.array([4, 0, 4, 0], np.int32)
    elif how == "doubled":
        for i in range(wl.n):
            a, b = int(wl.rect_off[i]), int(wl.rect_off[i + 1])
            size = r[a:b, 2:] - r[a:b, :2]
            for k in range(b - a):
                same = np.flatnonzero((size[:k] == size[k]).all(1))
                if len(same):
                    r[a + k] = r[a + same[0]]
    else:  # another set's
        r = np.roll(r, 3, axis=0)
    return np.ascontiguousarray(r, np.int32)


def _pairs(n):
    rng = np.random.default_rng(n)
    p = np.stack(np.meshgrid(np.arange(n), np.arange(n), indexing="ij"), -1).reshape(-1, 2)
    p = np.concatenate([p[rng.permutation(len(p))[:240]], [[n - 1, n - 1], [n - 2, n - 2], [n - 2, n - 1]]])
    return p[np.lexsort((p[:, 1], p[:, 0]))].astype(np.int32)


def _same_as_oracle(g, o):
    for f in ("dx_dbu", "dy_dbu", "pass_"):
        np.testing.assert_array_equal(g[f], o[f], err_msg=f)
    np.testing.assert_array_equal(g["score"].astype(np.int64), o["score"])
    assert np.abs(g["sim"].astype(np.float64) - o["sim"]).max() <= 1e-5


@pytest.mark.parametrize("how", ["mirrored", "moved", "doubled", "another"])
@pytest.mark.parametrize("px", [128, 256, 512])
def test_records_are_the_rasters(ctx, torch_cuda, px, how):
    import paper_2512_13133_gb300 as pcl
    wl = _workload(px)
    pairs = _pairs(wl.n)
    tp = torch_cuda.from_numpy(pairs).cuda()
    o = oracle.ClipSet(wl).match(pairs.astype(np.int64), oracle.MODE_COSINE, use_gates=False)
    engines = [pcl.ENGINE_FFT_PCM] if px == 512 else [pcl.ENGINE_EXACT_SCAN, pcl.ENGINE_TC_DIRECT,
                                                      pcl.ENGINE_TC_DIRECT_FP8]
    for e in engines:
        P = pcl.params(4 * px, 4, px // 4, cos_engine=e, flags=pcl.P_NO_GATES)
        cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
        pcl.pcl_rasterize(ctx, P, cs)
        cs.rects.copy_(torch_cuda.from_numpy(_rewritten(wl, how).reshape(-1)))
        _same_as_oracle(pcl.records_to_numpy(pcl.match(ctx, P, pcl.MODE_COSINE, cs, cs, tp)), o)
        if px == 512:
            work = np.zeros(len(pairs), pcl.WORK_DTYPE)
            work["a"], work["b"], work["mode"] = pairs[:, 0], pairs[:, 1], pcl.MODE_COSINE
            rec = torch_cuda.zeros((len(pairs), 40), dtype=torch_cuda.uint8, device="cuda")
            tw = torch_cuda.from_numpy(work.view(np.uint8).reshape(-1, 12)).cuda()
            pcl.pcl_match_mixed(ctx, [P], [cs], tw, len(pairs), rec)
            _same_as_oracle(pcl.records_to_numpy(rec), o)
