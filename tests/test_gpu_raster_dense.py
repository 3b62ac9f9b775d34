"""Clips of many rectangles: the order by area (ties by index) at the sizes around a
staged chunk and far past it, and a rasterisation time that grows about as the rectangles
do, not as their square."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _clips(rng, counts, W):
    out = []
    for k in counts:
        lo = rng.integers(0, W - 40, size=(k, 2))
        out.append(np.concatenate([lo, lo + rng.integers(1, 40, size=(k, 2))], 1))  # few areas: many ties
    return out


@pytest.mark.parametrize("px", [64, 128, 256, 512])
def test_order_by_area(torch, px):
    import paper_2512_13133_gb300 as pcl
    counts = [1, 31, 127, 128, 129, 255, 256, 257, 384, 385, 1000]
    clips = _clips(np.random.default_rng(px), counts, 4 * px)
    wl = synth.from_lists([c.tolist() for c in clips], 4 * px, 4, px // 4)
    P = pcl.params(4 * px, 4, px // 4)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(pcl.Context(0), P, cs)
    order = cs.rorder.cpu().numpy().view(np.uint16)
    for i, c in enumerate(clips):
        area = (c[:, 2] - c[:, 0]) * (c[:, 3] - c[:, 1])
        a, b = int(wl.rect_off[i]), int(wl.rect_off[i + 1])
        np.testing.assert_array_equal(order[a:b], np.argsort(area, kind="stable"), err_msg=f"{len(c)} rectangles")


def test_time_grows_with_the_rectangles(torch):
    """1,000 rectangles a clip take less than eight times 300 (the square: eleven times)"""
    import paper_2512_13133_gb300 as pcl
    ctx = pcl.Context(0)
    P = pcl.params(2048, 4, 128)
    times = {}
    for k in (300, 1000):
        c = _clips(np.random.default_rng(k), [k], 2048)[0]
        off = (np.arange(2001) * k).astype(np.uint32)
        cs = pcl.alloc_clipset(P, off, np.tile(c, (2000, 1)).astype(np.int32), with_spec=False)
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            pcl.pcl_rasterize(ctx, P, cs)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times[k] = best
    assert times[1000] < 8 * times[300], times
