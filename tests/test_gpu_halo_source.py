"""The halo rasters are what a re-extraction record is about: rectangles written again
after the rasters were made (mirrored, moved by a pixel, one doubled onto another
of its size, another set's, cut to the window) change no record, whether they are
the representatives' or the members'."""
import functools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _workload(px):
    W, m = 4 * px, px // 4
    wl = synth.generate(px + 1, n_clips=20, n_seeds=4, n_copies=12, window_dbu=W, margin_dbu=m, min_rects=2,
                        max_rects=max(4, px // 16), edge_jitter=3, halo_dbu=m)
    clips = [wl.clip(i).tolist() for i in range(wl.n)]
    s = W // 8  # two squares of one size; one that crosses the window's border
    clips += [[[s, s, 2 * s, 2 * s], [5 * s, 4 * s, 6 * s, 5 * s]], [[-m, s, m, 2 * s], [4 * s, 5 * s, 6 * s, 6 * s]]]
    return synth.from_lists(clips, W, 4, m)


def _rewritten(wl, how):
    r = wl.rects.reshape(-1, 4).copy()
    W = wl.window_dbu
    if how == "mirrored":
        r[:, [0, 2]] = W - r[:, [2, 0]]
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
    elif how == "cut":
        r = np.clip(r, 0, W)
    else:
        r = np.roll(r, 3, axis=0)
    return np.ascontiguousarray(r.reshape(-1), np.int32)


@functools.lru_cache(maxsize=None)
def _case(px):
    wl = _workload(px)
    pairs = np.stack(np.meshgrid(np.arange(wl.n), np.arange(wl.n), indexing="ij"), -1).reshape(-1, 2)
    pairs = pairs[np.random.default_rng(px).permutation(len(pairs))[:70 if px < 512 else 10]]
    pairs = np.concatenate([pairs, [[wl.n - 1, wl.n - 1], [wl.n - 2, wl.n - 2], [wl.n - 2, wl.n - 1], [0, 0]]])
    return wl, pairs, oracle.ClipSet(wl, halo=True).match(pairs.astype(np.int64), oracle.MODE_COSINE_HALO)


@pytest.mark.parametrize("side", ["representatives", "members"])
@pytest.mark.parametrize("how", ["mirrored", "moved", "doubled", "cut", "another"])
@pytest.mark.parametrize("px", [64, 256, 512])
def test_records_are_the_rasters(px, how, side):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    ctx = pcl.Context(0)
    wl, pairs, o = _case(px)
    P = pcl.params(4 * px, 4, px // 4)
    a, b = (pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False) for _ in range(2))
    pcl.pcl_rasterize(ctx, P, a)
    hb, nb = pcl.alloc_halo(P, b)
    pcl.pcl_rasterize_halo(ctx, P, b, hb, nb)
    (a if side == "representatives" else b).rects.copy_(torch.from_numpy(_rewritten(wl, how)))
    rec = torch.zeros((len(pairs), 40), dtype=torch.uint8, device="cuda")
    pcl.pcl_match_halo(ctx, P, a, b, hb, nb, torch.from_numpy(pairs.astype(np.int32)).cuda(), rec)
    g = pcl.records_to_numpy(rec)
    for f in ("dx_dbu", "dy_dbu", "pass_"):
        np.testing.assert_array_equal(g[f], o[f], err_msg=f)
    np.testing.assert_array_equal(g["score"].astype(np.int64), o["score"])
    np.testing.assert_array_equal(g["reserved"].astype(np.int64), o["pad"].astype(np.int64))
    assert np.abs(g["sim"].astype(np.float64) - o["sim"]).max() <= 1e-5
