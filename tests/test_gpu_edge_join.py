"""The self-join edge screen by bit tables (groups of 256 clips, four groups per
warp, tables of 64 groups at a time, one-CTA sort up to 8,192 clips): candidate
sets and gate counts equal the oracle's at the edges of those sizes, on layouts
with wires longer than the 16 cells one table reading covers, clips without
edges in an axis, rectangles past the window, empty clips and clips of more
than 64 polygons; beyond the oracle's reach they equal the union of the shards
(the tiled screen)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    return pcl.Context(0)


def _layouts(n, pitch, seed):
    """clips of W = 256 * pitch dbu: random rectangles, one in three with long wires, some special"""
    rng = np.random.default_rng(seed)
    W = 256 * pitch
    base = synth.generate(seed, n_clips=n, n_seeds=max(1, n // 8), n_copies=n // 2, window_dbu=W, margin_dbu=16 * pitch,
                          min_rects=1, max_rects=12, pitch_dbu=pitch)
    clips = []
    for i in range(n):
        c = base.clip(i).tolist()
        if i % 3 == 0:
            y = int(rng.integers(0, W - 40))
            c.append([int(rng.integers(0, W // 3)), y, int(rng.integers(W // 2, W + 1)), y + int(rng.integers(8, 40))])
        if i % 11 == 5:  # the whole width: no x edges off the border
            y = int(rng.integers(0, W - 100))
            c = [[0, y, W, y + 64]]
        if i % 17 == 3:
            c = [[-24, 40, 80, 120], [W // 2, W - 60, W // 2 + 90, W + 30]]
        if i % 29 == 7:
            c = []
        if i % 97 == 13:
            c = [[20 + 24 * (k % 10), 20 + 24 * (k // 10), 32 + 24 * (k % 10), 32 + 24 * (k // 10)]
                 for k in range(66 + i % 3)]
        clips.append(c)
    return synth.from_lists(clips, W, pitch, 16 * pitch)


def _clipset(ctx, wl, tol):
    import paper_2512_13133_gb300 as pcl
    P = pcl.params(wl.window_dbu, wl.pitch_dbu, wl.marker_dbu, edge_tol_dbu=tol)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    return P, cs


def _keys(pairs, n):
    return np.sort(pairs[:, 0].astype(np.int64) * n + pairs[:, 1])


@pytest.mark.parametrize("n,pitch", [(2, 4), (255, 4), (256, 3), (257, 4), (1025, 4), (1300, 3)])
def test_join_equals_oracle(ctx, n, pitch):
    import paper_2512_13133_gb300 as pcl
    wl = _layouts(n, pitch, n + pitch)
    P, cs = _clipset(ctx, wl, 6)
    gp, gc = pcl.candidates(ctx, P, pcl.MODE_EDGE, cs)
    op, oc = oracle.ClipSet(wl).candidates(pcl.MODE_EDGE, edge_tol_dbu=6)
    np.testing.assert_array_equal(_keys(gp.cpu().numpy(), n), _keys(op, n))
    np.testing.assert_array_equal(gc[:7], oc[:7].astype(np.int64))


@pytest.mark.parametrize("n", [8192, 8193, 16385, 33000])
def test_join_equals_union_of_shards(ctx, n):
    import paper_2512_13133_gb300 as pcl
    wl = _layouts(n, 4, n)
    P, cs = _clipset(ctx, wl, 4)
    gp, gc = pcl.candidates(ctx, P, pcl.MODE_EDGE, cs, cap=1 << 22)
    parts, counts = [], np.zeros(16, np.int64)
    for s in range(2):
        p, c = pcl.candidates(ctx, P, pcl.MODE_EDGE, cs, cap=1 << 22, shard=s, n_shards=2)
        parts.append(p.cpu().numpy())
        counts += c
    np.testing.assert_array_equal(_keys(gp.cpu().numpy(), n), _keys(np.concatenate(parts), n))
    np.testing.assert_array_equal(gc, counts)
