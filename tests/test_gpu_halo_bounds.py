"""The halo rasters and their tables (window counts of every shift, row and column
bounds) against their definitions, at markers from 0 to 32, a pitch that is no power
of two, clips of more than 128 rectangles, empty, full, sharing pixels and past
the halo."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("px,S,pitch", [(64, 0, 4), (64, 4, 4), (64, 32, 4), (128, 7, 6), (128, 16, 4), (256, 16, 4),
                                        (256, 31, 3), (512, 32, 4)])
def test_tables_equal_definitions(px, S, pitch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    W, M = px * pitch, S * pitch
    rng = np.random.default_rng(px + S)
    lo = rng.integers(-M - 9, W + M, size=(6, 40, 2))
    clips = [np.concatenate([q, q + rng.integers(1, W // 4, size=q.shape)], 1).tolist() for q in lo]
    small = rng.integers(-M, W + M, size=(300, 2))
    clips += [[], [[-M - 50, -M - 50, W + M + 50, W + M + 50]], np.concatenate([small, small + 11], 1).tolist()]
    wl = synth.from_lists(clips, W, pitch, M)
    P = pcl.params(W, pitch, M)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    ctx = pcl.Context(0)
    hb, nb = pcl.alloc_halo(P, cs)
    pcl.pcl_rasterize_halo(ctx, P, cs, hb, nb)
    n, NH, K = len(clips), px + 2 * S, 2 * S + 1
    words = (NH + 63) // 64
    bits = np.unpackbits(hb.cpu().numpy()[:8 * n * NH * words].reshape(n, NH, 8 * words), axis=2, bitorder="little")
    nrm = nb.cpu().numpy()[:4 * n * (K * K + 2 * NH)].view(np.uint32).reshape(n, -1)
    at = 2 * pitch * (np.arange(NH) - S) + pitch  # doubled pixel centres
    for c, rects in enumerate(clips):
        img = np.zeros((NH, NH), np.int64)
        for x0, y0, x1, y1 in rects:
            img[np.ix_((2 * y0 <= at) & (at < 2 * y1), (2 * x0 <= at) & (at < 2 * x1))] = 1
        np.testing.assert_array_equal(bits[c, :, :NH], img)
        assert not bits[c, :, NH:].any()
        sums = np.zeros((NH + 1, NH + 1), np.int64)
        sums[1:, 1:] = img.cumsum(0).cumsum(1)
        # the window of shift (dx, dy) starts at (S - dx, S - dy)
        o = S - np.arange(-S, S + 1)
        win = (sums[o + px][:, o + px] - sums[o][:, o + px] - sums[o + px][:, o] + sums[o][:, o])
        np.testing.assert_array_equal(nrm[c, :K * K].reshape(K, K), win)
        rows = np.concatenate([np.zeros((NH, 1), np.int64), img.cumsum(1)], 1)
        cols = np.concatenate([np.zeros((1, NH), np.int64), img.cumsum(0)], 0)
        np.testing.assert_array_equal(nrm[c, K * K:K * K + NH], (rows[:, o + px] - rows[:, o]).max(1))
        np.testing.assert_array_equal(nrm[c, K * K + NH:], (cols[o + px] - cols[o]).max(0))
