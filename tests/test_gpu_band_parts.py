"""The cosine band join with its bands shared by several warps (sets with fewer
representatives than the GPU has warps): candidates and gate counts equal the
oracle's on small sets, and those of the shards (whose bands are shared by
another number of warps) around the sizes where that number changes."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,px,against_oracle", [(2, 128, True), (9, 64, True), (700, 128, True), (600, 256, True),
                                                 (300, 512, True), (1216, 128, False), (1217, 64, False),
                                                 (1900, 256, False), (4864, 128, False), (4865, 128, False)])
def test_shared_bands(n, px, against_oracle):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    W = 4 * px
    wl = synth.generate(n + px, n_clips=n, n_seeds=max(1, n // 20), n_copies=n // 2, window_dbu=W, margin_dbu=W // 16,
                        min_rects=1, max_rects=10, edge_jitter=4, shift_max=W // 32)
    clips = [[] if k % 41 == 7 else wl.clip(k).tolist() for k in range(n)]
    wl = synth.from_lists(clips, W, 4, W // 16)
    ctx = pcl.Context(0)
    P = pcl.params(W, 4, W // 16)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)

    def keys(p):
        p = np.asarray(p).astype(np.int64)
        return np.sort(p[:, 0] * n + p[:, 1])

    got, gates = pcl.candidates(ctx, P, pcl.MODE_COSINE, cs)
    got = keys(got.cpu().numpy())
    if against_oracle:
        want, counts = oracle.ClipSet(wl).candidates(oracle.MODE_COSINE)
        np.testing.assert_array_equal(got, keys(want))
        np.testing.assert_array_equal(gates[:6], counts[:6].astype(np.int64))
    shards = [pcl.candidates(ctx, P, pcl.MODE_COSINE, cs, shard=s, n_shards=3) for s in range(3)]
    np.testing.assert_array_equal(got, np.sort(np.concatenate([keys(p.cpu().numpy()) for p, _ in shards])))
    np.testing.assert_array_equal(gates, sum(c for _, c in shards))
