"""The cosine self-join's density gate as a matrix product (256x256 and 512x512 px
from 2,048 clips): candidates and gate counts equal those of the band join's
shards (the path without the product) at the edges of the panels of 128
representatives and blocks of 256 members, at thresholds from 0.80 to 0.95,
with empty clips, and on sets of nearly identical clips, where the list of
pairs left overflows and the band join takes over."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    return pcl.Context(0)


def _check(ctx, wl, num, cap=1 << 22):
    import paper_2512_13133_gb300 as pcl
    P = pcl.params(wl.window_dbu, wl.pitch_dbu, wl.marker_dbu, cos_num=num)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    n = wl.n

    def keys(p):
        p = p.cpu().numpy().astype(np.int64)
        return np.sort(p[:, 0] * n + p[:, 1])

    got, gates = pcl.candidates(ctx, P, pcl.MODE_COSINE, cs, cap=cap)
    want, counts = [], np.zeros(16, np.int64)
    for s in range(2):
        p, c = pcl.candidates(ctx, P, pcl.MODE_COSINE, cs, cap=cap, shard=s, n_shards=2)
        want.append(keys(p))
        counts += c
    np.testing.assert_array_equal(keys(got), np.sort(np.concatenate(want)))
    np.testing.assert_array_equal(gates, counts)
    assert gates.sum() == n * (n - 1) // 2
    assert pcl.pcl_device_error(ctx) == 0
    return len(got), gates


@pytest.mark.parametrize("n,px,num", [(2048, 256, 95), (2049, 256, 80), (2303, 256, 90), (6000, 256, 95),
                                      (2177, 512, 80), (3000, 512, 95)])
def test_equals_band_join(ctx, n, px, num):
    W = 4 * px
    wl = synth.generate(n + num, n_clips=n, n_seeds=n // 20, n_copies=int(0.7 * n), window_dbu=W, margin_dbu=W // 16,
                        min_rects=2, max_rects=30, edge_jitter=4, shift_max=W // 32)
    clips = [[] if k % 501 == 77 else wl.clip(k).tolist() for k in range(n)]
    _check(ctx, synth.from_lists(clips, W, 4, W // 16), num)


def test_overflow_takes_the_band_join(ctx):
    n = 2500
    wl = synth.generate(5, n_clips=n, n_seeds=n // 20, n_copies=n // 2, window_dbu=1024, margin_dbu=64, min_rects=5,
                        max_rects=12)
    one = wl.clip(3).tolist()
    clips = [one if k % 10 else wl.clip(k).tolist() for k in range(n)]
    kept, _ = _check(ctx, synth.from_lists(clips, 1024, 4, 64), 95)
    assert kept > 2_000_000  # far more than the 65,536 listed pairs


@pytest.mark.parametrize("nq,nl,px,num", [(1, 2048, 256, 95), (129, 2300, 256, 80), (700, 5000, 256, 90),
                                          (300, 2100, 512, 80)])
def test_two_sets_equal_pairs_of_the_union(ctx, nq, nl, px, num):
    """queries x library through the product equal the cross pairs of the union's shards"""
    import paper_2512_13133_gb300 as pcl
    W, n = 4 * px, nq + nl
    wl = synth.generate(n + num, n_clips=n, n_seeds=n // 20, n_copies=int(0.7 * n), window_dbu=W, margin_dbu=W // 16,
                        min_rects=2, max_rects=30, edge_jitter=4, shift_max=W // 32)
    clips = [[] if k % 301 == 0 else wl.clip(k).tolist() for k in range(n)]
    wl = synth.from_lists(clips, W, 4, W // 16)
    P = pcl.params(W, 4, W // 16, cos_num=num)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    got, gates = pcl.candidates(ctx, P, pcl.MODE_COSINE, cs.view(P, 0, nq), b=cs.view(P, nq, n))
    got = got.cpu().numpy().astype(np.int64)
    want = np.concatenate([pcl.candidates(ctx, P, pcl.MODE_COSINE, cs, shard=s, n_shards=2)[0].cpu().numpy()
                           for s in range(2)]).astype(np.int64)
    want = want[(want[:, 0] < nq) & (want[:, 1] >= nq)]
    np.testing.assert_array_equal(np.sort(got[:, 0] * n + got[:, 1] + nq), np.sort(want[:, 0] * n + want[:, 1]))
    assert gates.sum() == nq * nl and gates[0] == len(got)


def test_wait_limit_takes_the_band_join(ctx):
    """a wait that runs out gives the product up; the result stays exact and no error is left"""
    import paper_2512_13133_gb300 as pcl
    wl = synth.generate(9, n_clips=3000, n_seeds=150, n_copies=2100, window_dbu=1024, margin_dbu=64, min_rects=3,
                        max_rects=20, edge_jitter=2)
    pcl.pcl_set_wait_limit(ctx, 1)
    try:
        _check(ctx, wl, 90)
    finally:
        pcl.pcl_set_wait_limit(ctx, 0)
    _check(ctx, wl, 90)
