// Cosine records from the clips' rectangles (rect_corr.cuh): the kernel in front
// of the exact window scan and of the tensor-core correlation, whose records it
// gives for every pair of clips with few enough rectangles that share no pixel.
#include "gates.cuh"
#include "rect_corr.cuh"

namespace pcl {

namespace {
using namespace rect_corr;

constexpr int kWarps = 4;

// The clips' verdicts (rect_corr.cuh), a warp per clip
__global__ void __launch_bounds__(32 * kWarps) rect_verdict_kernel(pcl_params prm, pcl_clipset cs, uint64_t base,
                                                                  uint64_t clips, uint64_t n,
                                                                  const unsigned long long *d_n, pcl_record *out) {
    if (d_n && *d_n < n) n = *d_n;
    if (!verdicts_pay(n, clips)) return;
    __shared__ short4 ranges[kWarps][kRectMax];
    const Geo g = make_geo(prm);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int psh = (g.p & (g.p - 1)) == 0 ? 31 - __clz(g.p) : -1;
    for (uint64_t c = (uint64_t)blockIdx.x * kWarps + warp; c < cs.n_clips; c += (uint64_t)gridDim.x * kWarps) {
        const bool ok = window_verdict(cs, (uint32_t)c, g, psh, ranges[warp], lane);
        if (lane == 0) *verdict_at(out, base + c) = ok ? 1 : 0;
    }
}

// One warp per pair (grid stride): indices, emptiness, gates, then the record
// from the rectangles.  A pair that does not take that path is left to the
// caller's next kernel: keep[t] = 1 (else 0), or without keep a record with
// flags = kRectPending.  stats: groups of shifts as pcl_stats_get counts them, a pair
// decided here counting as one.  CTAS: resident per SM, 8 (64 registers) where the
// tables of shifts leave room for them (100,000 pairs of 256x256 px with a look at the raster
// per pair: 1.16 -> 1.03 ms a call against 5), else 3 (12,001 of 512x512 px: 0.31 -> 0.26 ms
// against 8's registers).
template <int CTAS>
__global__ void __launch_bounds__(32 * kWarps, CTAS) rect_pair_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B,
                                                                      const pcl_pair *pairs, uint64_t n,
                                                                      const unsigned long long *d_n, pcl_record *out,
                                                                      uint32_t *keep, unsigned long long *stats,
                                                                      uint64_t clips) {
    if (d_n && *d_n < n) n = *d_n;
    const bool verdicts = clips && verdicts_pay(n, clips);
    extern __shared__ __align__(16) unsigned char smem[];
    const Geo g = make_geo(prm);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int psh = (g.p & (g.p - 1)) == 0 ? 31 - __clz(g.p) : -1;
    const Scratch s = scratch_at(smem + warp * scratch_bytes(g.S), g.S);
    const int K = 2 * g.S + 1;
    uint16_t *g2 = 4 * K * K >= 2 * kG2Scratch ? reinterpret_cast<uint16_t *>(s.table) : nullptr;
    const uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const bool rects = has_rects(A) && has_rects(B);
    unsigned long long done_here = 0;
    for (uint64_t t = w0; t < n; t += nw) {  // warp-uniform
        const pcl_pair pr = pairs[t];
        pcl_record rec{};
        rec.a = pr.a;
        rec.b = pr.b;
        rec.mode = PCL_MODE_COSINE;
        bool done = true, next = false;  // ends with rec, left to the next kernel
        if (pr.a >= A.n_clips || pr.b >= B.n_clips) {
            rec.flags = PCL_GATE_BAD_INDEX;
        } else {
            const uint32_t pa = A.pop[pr.a], pb = B.pop[pr.b];
            int gate = 0;
            if (pa == 0 && pb == 0) {
                rec.flags = PCL_F_EMPTY;
                rec.sim = 1.0f;
                rec.pass = 1;
            } else if (!(prm.flags & PCL_P_NO_GATES) &&
                       (gate = warp_cosine_gate(A, pr.a, B, pr.b, g, prm.cos_num, prm.cos_den, lane, g2)) != 0) {
                rec.flags = (uint16_t)gate;
            } else {
                done = false;
                next = !rects || pa == 0 || pb == 0 || 
                       !rect_record(prm, g, psh, A, B, pr, s, verdicts ? (int)out[t].reserved : -1, out + t, lane);
                done_here += next ? 0 : 1;
            }
        }
        if (lane == 0) {
            if (next && !keep) rec.flags = kRectPending;
            if (done || (next && !keep)) out[t] = rec;
            if (keep) keep[t] = next ? 1u : 0u;
        }
    }
    if (lane == 0 && stats && done_here) {
        atomicAdd(stats, done_here);
        atomicAdd(stats + 1, done_here * (unsigned long long)(K * (g.S / 8 + (g.S + 7) / 8 + 1)));
    }
}

}  // namespace

cudaError_t launch_rect_pairs(const pcl_params &prm, const pcl_clipset &a, const pcl_clipset &b, const pcl_pair *pairs,
                              uint64_t n, const unsigned long long *d_n, pcl_record *out, uint32_t *keep, int num_sms,
                              unsigned long long *stats, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const Geo g = make_geo(prm);
    const size_t sm = kWarps * scratch_bytes(g.S);
    auto *kern = 8 * sm <= 200 * 1024 ? rect_pair_kernel<8> : rect_pair_kernel<3>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kWarps, sm);
    if (e != cudaSuccess) return e;
    const uint64_t cap = (uint64_t)num_sms * (uint64_t)(per_sm > 0 ? per_sm : 1), need = (n + kWarps - 1) / kWarps;
    const bool one = one_set(a, b);
    uint64_t clips = (uint64_t)a.n_clips + (one ? 0 : b.n_clips);
    if (!has_rects(a) || !has_rects(b) || !verdicts_pay(n, clips)) clips = 0;
    if (clips) {
        const unsigned most = (unsigned)num_sms * 16;
        const uint64_t base_b = one ? 0 : a.n_clips;
        if (a.n_clips)
            rect_verdict_kernel<<<min((unsigned)(((uint64_t)a.n_clips + kWarps - 1) / kWarps), most), 32 * kWarps, 0, st>>>(
                prm, a, 0, clips, n, d_n, out);
        if (!one && b.n_clips)
            rect_verdict_kernel<<<min((unsigned)(((uint64_t)b.n_clips + kWarps - 1) / kWarps), most), 32 * kWarps, 0, st>>>(
                prm, b, base_b, clips, n, d_n, out);
        pair_verdict_kernel<<<(unsigned)((n + 255) / 256 < most ? (n + 255) / 256 : most), 256, 0, st>>>(
            a.n_clips, b.n_clips, base_b, clips, pairs, n, d_n, out);
    }
    kern<<<(unsigned)(need < cap ? need : cap), 32 * kWarps, sm, st>>>(prm, a, b, pairs, n, d_n, out, keep,
                                                                       stats, clips);
    return cudaGetLastError();
}

}  // namespace pcl
