"""What a served request counts of the memory budget: the tensor-core engine's
workspace is 20 bytes per candidate slot."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", ["f16", "bf16", "e4m3"])
def test_tensor_core_workspace_per_slot(engine):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_13133_gb300 as pcl
    wl = synth.generate(3, n_clips=300, n_seeds=20, n_copies=200, window_dbu=512, margin_dbu=32, min_rects=3,
                        max_rects=12, edge_jitter=3)
    q = synth.from_lists([wl.clip(k).tolist() for k in range(64)], 512, 4, 32)
    ctx = pcl.Context(0)
    tc = {"f16": pcl.ENGINE_TC_DIRECT, "bf16": pcl.ENGINE_TC_DIRECT_BF16, "e4m3": pcl.ENGINE_TC_DIRECT_FP8}[engine]
    used = {}
    for e in (tc, pcl.ENGINE_EXACT_SCAN):
        P = pcl.params(512, 4, 32, cos_engine=e)
        lib = pcl.alloc_clipset(P, wl.rect_off, wl.rects, with_spec=False)
        pcl.pcl_rasterize(ctx, P, lib)
        for slots in (20000, 40000):
            srv = pcl.Server(ctx, P, lib, max_inflight=1, max_query_clips=64, cand_per_query=slots, mem_budget=1 << 30)
            assert srv.submit(q.rect_off, q.rects, 1)
            used[e, slots] = (1 << 30) - srv.stats()[1]
            done = []
            while not done:
                done = srv.poll()
            assert done[0]["status"] == 0 and len(done[0]["pass_pairs"]) >= 64
            srv.close()
    x = pcl.ENGINE_EXACT_SCAN
    per_slot = ((used[tc, 40000] - used[tc, 20000]) - (used[x, 40000] - used[x, 20000])) / (64 * 20000)
    assert abs(per_slot - 20) < 0.01
