"""Gate counts of the edge self-join where all clips, or most, have one polygon count (one
bin of the bounding-box test), and the same pairs without counts asked for: equal to
the two shards of the tiled screen."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,polygons", [(2, [4]), (33, [3]), (700, [5]), (2500, [4]), (1500, [1, 1, 1, 2]), (300, [0, 2])])
def test_one_polygon_count(n, polygons):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    rng = np.random.default_rng(n)
    clips = []
    for i in range(n):
        r = []
        for k in range(polygons[i % len(polygons)]):  # a polygon per quarter strip, off the border but for some
            x, y = 130 * k + int(rng.integers(0, 30)), int(rng.integers(0, 400))
            r.append([x, y, x + int(rng.integers(20, 60)), y + int(rng.integers(20, 100))])
        clips.append(r)
    wl = synth.from_lists(clips, 1024, 4, 64)
    ctx = pcl.Context(0)
    P = pcl.params(1024, 4, 64)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    want, counts = [], 0
    for s in range(2):
        p, c = pcl.candidates(ctx, P, pcl.MODE_EDGE, cs, shard=s, n_shards=2)
        want.append(p.long())
        counts = counts + c
    want = torch.cat(want)
    want = torch.sort(want[:, 0] * n + want[:, 1]).values
    got, c = pcl.candidates(ctx, P, pcl.MODE_EDGE, cs)
    np.testing.assert_array_equal(c, counts)
    assert torch.equal(torch.sort(got[:, 0].long() * n + got[:, 1]).values, want)
    out = torch.zeros((max(1, len(want)), 2), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    pcl.pcl_candidates(ctx, P, pcl.MODE_EDGE, cs, out, cnt)
    assert int(cnt.item()) == len(want)
    assert len(want) == 0 or torch.equal(torch.sort(out[:, 0].long() * n + out[:, 1]).values, want)
