"""Records from the clips' rectangles (the kernel in front of the exact window scan,
the tensor-core engine, the mixed batch's 512x512 px class and re-extraction):
clips whose rectangles share pixels, clips of 64 and 65 rectangles, empty, full,
sub-pixel and out-of-window ones, beside plain clips and near copies, at markers
from 0 to N/16.  Shift, overlap, decision and similarity equal the oracle's, and
the tensor-core engine gives the same bytes when its own wait limit keeps every
pair on the tensor cores."""
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


def _workload(px, S, seed, halo=False):
    W = 4 * px
    m = 4 * S
    wl = synth.generate(seed, n_clips=24, n_seeds=4, n_copies=14, window_dbu=W, margin_dbu=m, min_rects=2,
                        max_rects=max(4, px // 16), edge_jitter=3, halo_dbu=m if halo else 0)
    clips = [wl.clip(i).tolist() for i in range(wl.n)]
    rng = np.random.default_rng(seed)
    side = W // 12

    def lattice(k):
        c = int(np.ceil(np.sqrt(k)))
        p = W // c
        return [[p * (i % c), p * (i // c), p * (i % c) + p // 2, p * (i // c) + p // 2] for i in range(k)]

    xy = rng.integers(0, W - side, size=(12, 2))
    clips += [[], [[0, 0, W, W]], [[W // 2, W // 2, W // 2 + 1, W // 2 + 1]], lattice(64), lattice(65),
              np.concatenate([xy, xy + side], 1).tolist(),  # sharing pixels
              [[20, 20, 120, 120], [20, 20, 120, 120]], [[-8, 30, 60, 90], [W - 40, W - 40, W + 8, W + 8]]]
    return synth.from_lists(clips, W, 4, m)


def _pairs(wl):
    n = wl.n
    rng = np.random.default_rng(n)
    p = np.stack(np.meshgrid(np.arange(n), np.arange(n), indexing="ij"), -1).reshape(-1, 2)
    p = p[rng.permutation(len(p))[:600]]
    return p[np.lexsort((p[:, 1], p[:, 0]))].astype(np.int32)


def _same_as_oracle(g, o):
    for f in ("dx_dbu", "dy_dbu", "pass_"):
        np.testing.assert_array_equal(g[f], o[f], err_msg=f)
    al = (o["flags"] & oracle.F_ALIGNED) > 0
    np.testing.assert_array_equal(g["score"][al].astype(np.int64), o["score"][al])
    assert np.abs(g["sim"].astype(np.float64) - o["sim"]).max() <= 1e-5


@pytest.mark.parametrize("px,S", [(64, 4), (128, 8), (128, 5), (256, 16), (256, 0), (256, 13), (512, 32), (512, 21)])
def test_records_equal_oracle(ctx, torch_cuda, px, S):
    import paper_2512_13133_gb300 as pcl
    wl = _workload(px, S, px + S)
    pairs = _pairs(wl)
    tp = torch_cuda.from_numpy(pairs).cuda()
    o = oracle.ClipSet(wl).match(pairs.astype(np.int64), oracle.MODE_COSINE, use_gates=False)
    engines = {64: [pcl.ENGINE_TC_DIRECT], 512: [pcl.ENGINE_FFT_PCM]}.get(
        px, [pcl.ENGINE_EXACT_SCAN, pcl.ENGINE_TC_DIRECT, pcl.ENGINE_TC_DIRECT_FP8])
    for e in engines:
        P = pcl.params(4 * px, 4, 4 * S, cos_engine=e, flags=pcl.P_NO_GATES)
        cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
        pcl.pcl_rasterize(ctx, P, cs)
        r = pcl.match(ctx, P, pcl.MODE_COSINE, cs, cs, tp)
        _same_as_oracle(pcl.records_to_numpy(r), o)
        if e in (pcl.ENGINE_TC_DIRECT, pcl.ENGINE_TC_DIRECT_FP8):
            pcl.pcl_set_wait_limit(ctx, 1_000_000_000)
            plain = pcl.match(ctx, P, pcl.MODE_COSINE, cs, cs, tp)
            pcl.pcl_set_wait_limit(ctx, 0)
            assert pcl.pcl_device_error(ctx) == 0
            assert torch_cuda.equal(r, plain)


@pytest.mark.parametrize("px,S", [(64, 4), (128, 8), (256, 16), (256, 9), (512, 32)])
def test_halo_records_equal_oracle(ctx, torch_cuda, px, S):
    import paper_2512_13133_gb300 as pcl
    wl = _workload(px, S, 7 * px + S, halo=True)
    pairs = _pairs(wl)
    P = pcl.params(4 * px, 4, 4 * S)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    hb, nb = pcl.alloc_halo(P, cs)
    pcl.pcl_rasterize_halo(ctx, P, cs, hb, nb)
    rec = torch_cuda.zeros((len(pairs), 40), dtype=torch_cuda.uint8, device="cuda")
    pcl.pcl_match_halo(ctx, P, cs, cs, hb, nb, torch_cuda.from_numpy(pairs).cuda(), rec)
    o = oracle.ClipSet(wl, halo=True).match(pairs.astype(np.int64), oracle.MODE_COSINE_HALO)
    _same_as_oracle(pcl.records_to_numpy(rec), o)
