"""Candidate calls at the limits of their memory: a self-join captured with the
workspace of the general path alone (no allocation may happen in a capture)
takes that path with the same result, and the density gate's buffers of a
served request take nothing from the memory budget that admission counts."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _set(pcl, ctx, n, px=256):
    W = 4 * px
    wl = synth.generate(n, n_clips=n, n_seeds=n // 20, n_copies=int(0.7 * n), window_dbu=W, margin_dbu=W // 16,
                        min_rects=3, max_rects=20, edge_jitter=3)
    P = pcl.params(W, 4, W // 16, cos_engine=pcl.ENGINE_EXACT_SCAN)
    cs = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
    pcl.pcl_rasterize(ctx, P, cs)
    return wl, P, cs


@pytest.mark.parametrize("mode,n", [("edge", 700), ("cosine", 2100)])
def test_capture_with_the_general_workspace(torch_cuda, mode, n):
    import paper_2512_13133_gb300 as pcl
    torch = torch_cuda
    ctx = pcl.Context(0)
    _, P, cs = _set(pcl, ctx, n)
    m = pcl.MODE_EDGE if mode == "edge" else pcl.MODE_COSINE
    want, counts = pcl.candidates(pcl.Context(0), P, m, cs)
    if mode == "edge":
        pcl.candidates(ctx, P, m, cs, b=cs)  # grows the context workspace to the pair list
    else:
        pcl.candidates(ctx, P, m, cs, shard=0, n_shards=2)  # to the area order
    out = torch.zeros((1 << 20, 2), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    gates = torch.zeros(16, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pcl.pcl_candidates(ctx, P, m, cs, out, cnt, gates)
    graph.replay()
    torch.cuda.synchronize()
    got = out[:int(cnt.item())].long()
    key = torch.sort(got[:, 0] * n + got[:, 1]).values
    assert torch.equal(key, torch.sort(want[:, 0].long() * n + want[:, 1]).values)
    np.testing.assert_array_equal(gates.cpu().numpy(), counts)


def test_admission_takes_no_product_buffers(torch_cuda):
    import paper_2512_13133_gb300 as pcl
    ctx = pcl.Context(0)
    wl, P, cs = _set(pcl, ctx, 2400)
    q = synth.from_lists([wl.clip(k).tolist() for k in range(64)], wl.window_dbu, 4, wl.marker_dbu)

    def serve(n_lib, budget, requests=1):
        srv = pcl.Server(ctx, P, cs.view(P, 0, n_lib), max_inflight=8, max_query_clips=64, cand_per_query=64,
                         mem_budget=budget)
        admitted = sum(srv.submit(q.rect_off, q.rects, i) for i in range(requests))
        used = budget - srv.stats()[1]
        done = {}
        while len(done) < admitted:
            done.update({c["id"]: c for c in srv.poll()})
        assert all(c["status"] == 0 for c in done.values())
        rec = [np.sort(c["records"], order=["a", "b"]) for c in done.values()]
        srv.close()
        return admitted, used, rec

    _, plain, _ = serve(2047, 1 << 28)  # no product below 2,048 clips
    _, used, with_product = serve(2400, 1 << 28)
    assert abs(used - plain) <= 4096  # the library's chunk counters
    admitted, _, _ = serve(2400, 3 * used + 256, requests=5)
    assert admitted == 3
    # a budget with no room for the product's buffers: the band join, same records
    _, _, without = serve(2400, used)
    np.testing.assert_array_equal(with_product[0][["a", "b", "score", "pass_"]], without[0][["a", "b", "score", "pass_"]])
