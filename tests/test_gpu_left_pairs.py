"""Pairs that the rectangle kernels leave to the scans (clips of more than 64
rectangles, or sharing pixels) beside pairs that they decide, in lists from one pair
to several rounds of the scans' grid, whole and cut short on the device: records
equal the oracle's, and a short list of such pairs is spread over the GPU."""
import functools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pcl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    return pcl


def _dense(rng, k, W, m):
    """k rectangles on a jittered lattice over [-m, W + m)"""
    c = int(np.ceil(np.sqrt(k)))
    p = (W + 2 * m) // c
    i = rng.permutation(c * c)[:k]
    j = rng.integers(0, p // 3, size=(k, 4))
    x, y = (i % c) * p - m, (i // c) * p - m
    return np.stack([x + j[:, 0], y + j[:, 1], x + p - 1 - j[:, 2], y + p - 1 - j[:, 3]], 1)


@functools.lru_cache(maxsize=None)
def _case(px, halo):
    W, m, n_pairs = 4 * px, px // 4, {128: 160, 256: 60, 512: 16}[px]
    h = m if halo else 0
    rng = np.random.default_rng(px + halo)
    base = [_dense(rng, k, W, h) for k in (65, 90, 12, 130, 64)]
    base.append(np.concatenate([base[2], base[2] + 9]))  # sharing pixels
    clips = [base[i % 6] + rng.integers(-m, m + 1) * (i >= 6) for i in range(36)]
    wl = synth.from_lists([(c if halo else np.clip(c, 0, W)).tolist() for c in clips], W, 4, m)
    pairs = np.concatenate([rng.integers(0, 36, size=(n_pairs // 2, 2)),
                            rng.integers(0, 6, size=(n_pairs - n_pairs // 2, 1)) + 6 * rng.integers(0, 6, size=(1, 2))])
    o = oracle.ClipSet(wl, halo=True).match(pairs, oracle.MODE_COSINE_HALO) if halo else \
        oracle.ClipSet(wl).match(pairs, oracle.MODE_COSINE, use_gates=False)
    return wl, pairs, o


def _caller(pcl, ctx, wl, halo):
    P = pcl.params(wl.window_dbu, 4, wl.marker_dbu, flags=pcl.P_NO_GATES,
                   cos_engine=pcl.ENGINE_FFT_PCM if halo or wl.raster_n == 512 else pcl.ENGINE_EXACT_SCAN)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    if not halo:
        return lambda tp, rec, d_n=None: pcl.pcl_match_pairs(ctx, P, pcl.MODE_COSINE, cs, cs, tp, rec, d_n=d_n)
    hb, nb = pcl.alloc_halo(P, cs)
    pcl.pcl_rasterize_halo(ctx, P, cs, hb, nb)
    return lambda tp, rec, d_n=None: pcl.pcl_match_halo(ctx, P, cs, cs, hb, nb, tp, rec, d_n=d_n)


@pytest.mark.parametrize("halo", [False, True])
@pytest.mark.parametrize("px,n", [(128, 1), (128, 127), (128, 3001), (128, 200003), (256, 500), (256, 20000), (512, 700)])
def test_records_equal_oracle(pcl, px, n, halo):
    import torch
    wl, pairs, o = _case(px, halo)
    ctx = pcl.Context(0)
    call = _caller(pcl, ctx, wl, halo)
    pick = np.random.default_rng(n).integers(0, len(pairs), size=n)
    tp = torch.from_numpy(pairs[pick].astype(np.int32)).cuda()
    for count in {n, n - n // 3}:
        rec = torch.zeros((n, 40), dtype=torch.uint8, device="cuda")
        call(tp, rec, d_n=torch.tensor([count], dtype=torch.int64, device="cuda") if count < n else None)
        g = pcl.records_to_numpy(rec)
        assert not rec[count:].any()
        g, e = g[:count], o[pick[:count]]
        for f in ("dx_dbu", "dy_dbu", "pass_"):
            np.testing.assert_array_equal(g[f], e[f], err_msg=f)
        np.testing.assert_array_equal(g["score"].astype(np.int64), e["score"])
        assert np.abs(g["sim"].astype(np.float64) - e["sim"]).max() <= 1e-5


@pytest.mark.parametrize("halo", [False, True])
def test_short_lists_use_the_whole_gpu(pcl, halo):
    """64 pairs of dense clips take no longer than a few times one of them
    (one CTA after the other: 30 to 40 times)"""
    import torch
    wl, _, _ = _case(256, halo)
    ctx = pcl.Context(0)
    call = _caller(pcl, ctx, wl, halo)
    times = {}
    for n in (1, 64):
        tp = torch.tensor([[1, 7]] * n, dtype=torch.int32, device="cuda")
        rec = torch.zeros((n, 40), dtype=torch.uint8, device="cuda")
        best = float("inf")
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call(tp, rec)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times[n] = best
    assert times[64] < 6 * times[1], times
