"""Rasters and signatures of clips whose rectangles share pixels (column and block
counts are then counted from the rows) and of clips without (sums over the
rectangles), beside rectangles past the window, empty and sub-pixel ones, more
rectangles than a staged chunk and a pitch that is not a power of two: every
array equals its definition."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _clips(px, pitch, rng):
    W = px * pitch
    clips = [[], [[0, 0, W, W]], [[W // 2, W // 2, W // 2 + 1, W // 2 + 1]]]
    for k in range(24):
        n = [3, 40, 300][k % 3] if px >= 128 else [3, 20, 300][k % 3]
        side = W // 3 if k % 2 else max(W // 40, 2)
        xy = rng.integers(-side, W, size=(n, 2))
        wh = rng.integers(1, side + 1, size=(n, 2))
        r = np.concatenate([xy, xy + wh], 1)
        if k % 4 < 2:
            r = np.concatenate([np.clip(r[:, :2], 0, W - 1), np.clip(r[:, 2:], 1, W)], 1)
            r = r[(r[:, 0] < r[:, 2]) & (r[:, 1] < r[:, 3])]
        clips.append(r.tolist())
    clips.append([[8 * k, 8 * j, 8 * k + 4, 8 * j + 4] for k in range(W // 16) for j in range(W // 64)])  # a lattice
    return clips


@pytest.mark.parametrize("px,pitch", [(64, 4), (128, 4), (256, 3), (256, 4), (512, 4)])
def test_raster_definition(px, pitch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    clips = _clips(px, pitch, np.random.default_rng(px + pitch))
    W = px * pitch
    wl = synth.from_lists(clips, W, pitch, W // 16)
    P = pcl.params(W, pitch, W // 16 // pitch * pitch)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(pcl.Context(0), P, cs)
    got, sig = pcl.unpack_bits(cs), pcl.signatures(cs)
    at = 2 * pitch * np.arange(px) + pitch
    order = cs.rorder.cpu().numpy().view(np.uint16)
    occ = np.unpackbits(cs.occ.cpu().numpy()[:512 * wl.n].reshape(wl.n, 64, 8), axis=2, bitorder="little")
    rb = (cs.S + 15) // 16
    for i, rects in enumerate(clips):
        img = np.zeros((px, px), bool)
        grid = np.zeros((64, 64), bool)
        cell = W // 64
        for x0, y0, x1, y1 in rects:
            img |= ((2 * y0 <= at) & (at < 2 * y1))[:, None] & ((2 * x0 <= at) & (at < 2 * x1))[None]
            c = np.clip(np.array([x0, y0, x1 - 1, y1 - 1]) // cell, 0, 63)
            grid[c[1]:c[3] + 1, c[0]:c[2] + 1] = True
        np.testing.assert_array_equal(got[i], img)
        assert sig["pop"][i] == img.sum()
        np.testing.assert_array_equal(sig["rows"][i], img.sum(1))
        np.testing.assert_array_equal(sig["cols"][i], img.sum(0))
        blk = img.reshape(px // 16, 16, px // 16, 16).sum((1, 3))
        np.testing.assert_array_equal(sig["blk"][i], blk)
        p = np.pad(blk, rb)
        nb = px // 16
        dil = sum(p[a:a + nb, b:b + nb] for a in range(2 * rb + 1) for b in range(2 * rb + 1))
        np.testing.assert_array_equal(sig["dil"][i], np.minimum(dil, 65535))
        np.testing.assert_array_equal(occ[i], grid)
        area = [(r[2] - r[0]) * (r[3] - r[1]) for r in rects]
        np.testing.assert_array_equal(order[wl.rect_off[i]:wl.rect_off[i + 1]], np.argsort(area, kind="stable"))
