"""Candidates without allocation where the fixed scratch holds the density gate's matrix
product (from 2,048 clips of 256x256 and 512x512 px on) and just past it, at the default
wait limit and at one that runs out at once: the pairs and gate counts of the band
join alone (two shards)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit", [0, 1])
@pytest.mark.parametrize("px,n", [(256, 2047), (256, 2048), (256, 3400), (256, 3600), (512, 2100)])
def test_same_as_two_shards(px, n, limit):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    W = 4 * px
    wl = synth.generate(n, n_clips=n, n_seeds=n // 20, n_copies=int(0.7 * n), window_dbu=W, margin_dbu=W // 16,
                        min_rects=3, max_rects=20, edge_jitter=3)
    ctx = pcl.Context(0)
    P = pcl.params(W, 4, W // 16)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    want, counts = [], 0
    for s in range(2):
        p, c = pcl.candidates(ctx, P, pcl.MODE_COSINE, cs, shard=s, n_shards=2)
        want.append(p.long())
        counts = counts + c
    want = torch.cat(want)
    out = torch.zeros((1 << 20, 2), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    gates = torch.zeros(16, dtype=torch.int64, device="cuda")
    pcl.pcl_set_wait_limit(ctx, limit)
    pcl.pcl_candidates_cosine_noalloc(ctx, P, cs, out, cnt, gates)
    got = out[:int(cnt.item())].long()
    assert torch.equal(torch.sort(got[:, 0] * n + got[:, 1]).values, torch.sort(want[:, 0] * n + want[:, 1]).values)
    np.testing.assert_array_equal(gates.cpu().numpy(), counts)
