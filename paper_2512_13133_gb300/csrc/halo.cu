// Cosine matching with re-extraction of the member's window (Sec. 2.1: a
// pattern is the layout cut out around its centre, and the centre may lie
// anywhere in the marker region; Eq. 2 at every shift).
//
// Each clip carries its rectangles over [-M, W + M)^2.  Its halo raster
// samples that region at the pixel centres p i + p/2, i in [-S, N + S): row
// j + S, bit i + S of a row of NWH = ceil((N + 2S) / 64) words.  For the
// shift s the member's window moved by s holds the halo pixels x - s,
// x in [0, N)^2, so
//   c(s)   = sum_x A(x) Bh(x - s)         (A: the representative's window)
//   n_B(s) = sum_x Bh(x - s)              (pixels of the moved window)
//   sim(s) = c(s) / sqrt(|A| n_B(s)).
// n_B depends on the member alone: halo_raster_kernel tabulates it for every
// shift once per clip (the window sums of the halo raster, as a summed-area
// table would give them), beside the halo raster itself.  halo_pair_kernel
// counts c(s) by AND + popcount with both rasters staged in shared memory, each
// segment of equal row pairs once (row_segments in exact_dev.cuh; 60,000
// same-seed pairs of 256^2 px: 11.9 -> 8.3 ms), and keeps the shift of largest sim, compared exactly as
// c1^2 n2 vs c2^2 n1 (|A| is common; products < 2^55 up to 512^2 px), ties by
// smaller |dx| + |dy|, then dy, then dx; the decision is Eq. 2's exact rule
// with n_B(s*) for |B|.  No lossless gates here: they bound c against fixed
// norms.
#include "ctx.h"
#include "exact_dev.cuh"
#include "rect_corr.cuh"

using pcl::cos_exceeds;
using pcl::Geo;
using pcl::make_geo;

namespace {

constexpr int kThreads = 256;

__host__ __device__ inline int halo_side(int N, int S) { return N + 2 * S; }
__host__ __device__ inline int halo_words(int N, int S) { return (N + 2 * S + 63) / 64; }
// u32 per clip in the norms buffer: n_B(s) for the K^2 shifts, then the row
// bounds hrow[NH] and the column bounds hcol[NH] of the pair kernel's pruning
__host__ __device__ inline int norms_stride(int N, int S) { return (2 * S + 1) * (2 * S + 1) + 2 * halo_side(N, S); }

// shared-memory row strides in 64-bit words, odd so that the 16 lanes of a
// half-warp reading 16 consecutive rows hit 16 different bank pairs: A's rows
// (NW words) and the halo rows (NWH words and a zero word)
__host__ __device__ inline int a_stride(int NW) { return NW | 1; }
__host__ __device__ inline int h_stride(int NWH) { return (NWH + 1) | 1; }

// One CTA per clip: halo raster rows, the window sums n_B(s), and the pair
// kernel's bounds.  Bound by issue slots.  The rows' bits are set with a lane per rectangle.
// A window that moves by one takes one row (column) of ones in and leaves one
// out, so nothing is summed again for another shift: a thread slides along a row for its counts at
// every dx, a warp along 32 columns (transposed 32 rows at a time) for the
// column bound, and the sums over the rows at dy = -S are followed by prefix sums
// of what enters and leaves up to dy = S.  12,200 clips of 256x256 px and S = 16:
// about 200 us against 1,346 with every row testing every rectangle and each shift
// summed for itself.
constexpr int kRasterThreads = 288;  // nine warps: the rows and the column words of 256x256 px with S = 16
constexpr int kRectChunk = 128;      // rectangles staged at a time

__host__ __device__ inline int row_stride(int NWH) { return (2 * NWH) | 1; }  // 32-bit words of a row, odd
__host__ __device__ inline int cnt_stride(int NH) { return (NH + 1) & ~1; }

__global__ void __launch_bounds__(kRasterThreads) halo_raster_kernel(pcl_params prm, pcl_clipset cs, uint64_t *hbits,
                                                                     uint32_t *norms) {
    const Geo g = make_geo(prm);
    const int N = g.N, S = g.S, NH = halo_side(N, S), NWH = halo_words(N, S), K = 2 * S + 1;
    const int RS = row_stride(NWH), CS = cnt_stride(NH);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int T = kRasterThreads, W = T / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *rows = reinterpret_cast<uint32_t *>(smem);              // [NH][RS]
    uint32_t *nb_s = rows + (size_t)NH * RS;                          // [K][K] n_B, dy by dy
    uint16_t *cnt = reinterpret_cast<uint16_t *>(nb_s + (size_t)K * K);  // [K][CS] ones of each row in the window at dx
    __shared__ short4 rs[kRectChunk];  // pixel ranges {x0, x1, y0, y1} in the halo raster
    const uint32_t c = blockIdx.x;
    const int psh = (g.p & (g.p - 1)) == 0 ? 31 - __clz(g.p) : -1;
    const int32_t *r = cs.rects + 4 * (size_t)cs.rect_off[c];
    const int nr = (int)(cs.rect_off[c + 1] - cs.rect_off[c]);
    for (int t = tid; t < NH * RS; t += T) rows[t] = 0u;
    for (int base = 0; base < nr; base += kRectChunk) {
        const int n = min(kRectChunk, nr - base);
        __syncthreads();
        if (tid < n) {
            const int32_t *q = r + 4 * (size_t)(base + tid);
            auto at = [&](int v) { return (short)(pcl::rect_corr::pix_index(v, g.p, psh, -S, N + S) + S); };
            rs[tid] = make_short4(at(q[0]), at(q[2]), at(q[1]), at(q[3]));
        }
        __syncthreads();
        for (int t = lane; t < n; t += 32) {
            const short4 q = rs[t];
            if (q.x >= q.y) continue;
            const int w0 = q.x >> 5, w1 = (q.y - 1) >> 5;
            const uint32_t first = 0xffffffffu << (q.x & 31), last = 0xffffffffu >> (31 - ((q.y - 1) & 31));
            for (int j = q.z + warp; j < q.w; j += W) {
                uint32_t *row = rows + (size_t)j * RS;
                if (w0 == w1) {
                    atomicOr(row + w0, first & last);
                } else {
                    atomicOr(row + w0, first);
                    for (int w = w0 + 1; w < w1; ++w) atomicOr(row + w, 0xffffffffu);
                    atomicOr(row + w1, last);
                }
            }
        }
    }
    __syncthreads();
    uint32_t *nrm = norms + (size_t)c * norms_stride(N, S);
    for (int t = tid; t < NH * NWH; t += T) {
        const uint32_t *w = rows + (size_t)(t / NWH) * RS + 2 * (t % NWH);
        hbits[(size_t)c * NH * NWH + t] = (uint64_t)w[0] | ((uint64_t)w[1] << 32);
    }
    // rows: cnt[dx + S][t], the bits of halo row t at [S - dx, S - dx + N), and
    // their largest over dx.  From dx - 1 to dx bit S - dx enters, bit S - dx + N leaves.
    for (int t = tid; t < NH; t += T) {
        const uint32_t *w = rows + (size_t)t * RS;
        int n = 0;
        for (int k = 0; k < 2 * NWH; ++k) n += __popc(w[k]);
        uint64_t lo = 0, hi = 0;  // bits [0, 2S) and [N, N + 2S)
        if (S > 0) {
            lo = ((uint64_t)w[0] | ((uint64_t)w[1] << 32)) & (~0ull >> (64 - 2 * S));
            hi = (uint64_t)w[2 * g.nw] | ((uint64_t)w[2 * g.nw + 1] << 32);
        }
        n -= __popcll(lo);
        int m = n;
        cnt[t] = (uint16_t)n;
        for (int k = 1; k < K; ++k) {
            const int j = 2 * S - k;
            n += (int)((lo >> j) & 1u) - (int)((hi >> j) & 1u);
            m = max(m, n);
            cnt[(size_t)k * CS + t] = (uint16_t)n;
        }
        nrm[K * K + t] = (uint32_t)m;
    }
    // columns, 32 per warp: the most ones halo column x has in N rows [t0, t0 + N), t0 = 0 .. 2S
    for (int w = warp; w < 2 * NWH; w += W) {
        int n = 0;
        uint64_t lo = 0, hi = 0;  // this lane's column: rows [0, 64) and [N, N + 64)
        for (int b = 0; 32 * b < NH; ++b) {
            const int t = 32 * b + lane;
            const uint32_t col = pcl::transpose32(t < NH ? rows[(size_t)t * RS + w] : 0u, lane);
            if (b < 2) lo |= (uint64_t)col << (32 * b);
            if (32 * b < N) n += __popc(col);
            else hi |= (uint64_t)col << (32 * b - N);
        }
        int m = n;
        for (int j = 0; j < 2 * S; ++j) {
            n += (int)((hi >> j) & 1u) - (int)((lo >> j) & 1u);
            m = max(m, n);
        }
        if (32 * w + lane < NH) nrm[K * K + NH + 32 * w + lane] = (uint32_t)m;
    }
    __syncthreads();
    // n_B(dx, dy) = sum over the rows t in [S - dy, S - dy + N) of cnt, a warp per dx:
    // from dy - 1 to dy row S - dy enters, row S - dy + N leaves
    for (int k = warp; k < K; k += W) {
        const uint16_t *ck = cnt + (size_t)k * CS;
        int sum = 0;
        for (int t = lane; t < N; t += 32) sum += ck[2 * S + t];
        sum = __reduce_add_sync(0xffffffffu, sum);  // dy = -S
        if (lane == 0) nb_s[k] = (uint32_t)sum;
        for (int i0 = 0; i0 < 2 * S; i0 += 32) {
            const int t = 2 * S - 1 - (i0 + lane);
            int v = t >= 0 ? (int)ck[t] - (int)ck[t + N] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            if (t >= 0) nb_s[(size_t)(i0 + lane + 1) * K + k] = (uint32_t)(sum + v);
            sum += __shfl_sync(0xffffffffu, v, 31);
        }
    }
    __syncthreads();
    for (int t = tid; t < K * K; t += T) nrm[t] = nb_s[t];
}

// c for 8 shifts of one row pair: A's 32-bit word w against halo bits
// [32 (w + QQ) + r, +32), r = rb + u
template <int NW32, int QQ>
__device__ __forceinline__ void halo_row_counts(const uint32_t (&a)[NW32], const uint32_t (&h)[NW32 + 4], int rb,
                                                uint32_t times, uint32_t (&cnt)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int r = rb + u;
        uint32_t x[NW32];
#pragma unroll
        for (int w = 0; w < NW32; ++w) x[w] = a[w] & __funnelshift_r(h[w + QQ], h[w + QQ + 1], r);
        cnt[u] += times * pcl::popc_sum<NW32>(x);
    }
}

// row_starts (exact_dev.cuh) for rows of nw 64-bit words at stride sw
__device__ __forceinline__ void row_starts64(const uint64_t *rows, int n_rows, int nw, int sw, uint32_t *starts) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int w = warp; w < (n_rows + 31) / 32; w += nwarps) {
        const int y = 32 * w + lane;
        bool diff = y == 0;
        if (y > 0 && y < n_rows)
            for (int v = 0; v < nw && !diff; ++v) diff = rows[y * sw + v] != rows[(y - 1) * sw + v];
        const uint32_t m = __ballot_sync(0xffffffffu, diff);
        if (lane == 0) starts[w] = m;
    }
}

// sim(c1, n1) > sim(c2, n2), with |A| = pa common to both
__device__ __forceinline__ int sim_cmp(uint32_t c1, uint32_t n1, uint32_t c2, uint32_t n2, uint64_t pa) {
    uint64_t a1, d1, a2, d2;
    if (pa == 0 || n1 == 0) {
        a1 = (pa == 0 && n1 == 0) ? 1u : 0u;
        d1 = 1;
    } else {
        a1 = (uint64_t)c1 * c1;
        d1 = n1;
    }
    if (pa == 0 || n2 == 0) {
        a2 = (pa == 0 && n2 == 0) ? 1u : 0u;
        d2 = 1;
    } else {
        a2 = (uint64_t)c2 * c2;
        d2 = n2;
    }
    const uint64_t l = a1 * d2, r = a2 * d1;
    return l > r ? 1 : (l < r ? -1 : 0);
}

struct Best {
    uint32_t c, n;
    int dx, dy;
    bool valid;
};

// b1 before b2 in the order (-sim, |dx| + |dy|, dy, dx)
__device__ __forceinline__ bool before(const Best &b1, const Best &b2, uint64_t pa) {
    if (!b2.valid) return b1.valid;
    if (!b1.valid) return false;
    const int s = sim_cmp(b1.c, b1.n, b2.c, b2.n, pa);
    if (s) return s > 0;
    const int l1 = abs(b1.dx) + abs(b1.dy), l2 = abs(b2.dx) + abs(b2.dy);
    if (l1 != l2) return l1 < l2;
    if (b1.dy != b2.dy) return b1.dy < b2.dy;
    return b1.dx < b2.dx;
}

// the record of the pair's best shift
__device__ __forceinline__ pcl_record halo_record(const pcl_params &prm, const Geo &g, const pcl_pair pr, uint64_t pa,
                                                  const Best &b) {
    pcl_record rec{};
    rec.a = pr.a;
    rec.b = pr.b;
    rec.mode = PCL_MODE_COSINE;
    rec.dx_dbu = b.dx * g.p;
    rec.dy_dbu = b.dy * g.p;
    rec.score = b.c;
    rec.reserved = b.n;
    uint16_t fl = PCL_F_ALIGNED;
    float sim = 0.0f;
    if (pa == 0 && b.n == 0) {
        sim = 1.0f;
        rec.pass = 1;
        fl |= PCL_F_EMPTY;
    } else if (pa && b.n) {
        sim = (float)b.c / sqrtf((float)pa * (float)b.n);
        const float T = (float)prm.cos_num / (float)prm.cos_den;
        if (fabsf(sim - T) < prm.near_band) {
            fl |= PCL_F_NEAR_BAND;
            sim = (float)((double)b.c / sqrt((double)pa * (double)b.n));
        }
        rec.pass = cos_exceeds(b.c, pa, b.n, prm.cos_num, prm.cos_den) ? 1 : 0;
    }
    rec.sim = sim;
    rec.flags = fl;
    return rec;
}

// The n staged ranges are clip b's halo raster (hb) and share no pixel: every
// pixel of theirs is set, and the windows of the four corner shifts, which
// together cover the halo (2 S <= N), hold as many of them as tabulated (gn).
__device__ __forceinline__ bool ranges_are_halo(const short4 *r, int n, const uint64_t *__restrict__ hb,
                                                const uint32_t *__restrict__ gn, const Geo &g, int lane) {
    const int N = g.N, S = g.S, K = 2 * S + 1;
    uint32_t c[4] = {0u, 0u, 0u, 0u};
    for (int t = lane; t < n; t += 32) {
        const short4 q = r[t];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int dx = k & 1 ? S : -S, dy = k & 2 ? S : -S;  // the window starts at (-dx, -dy)
            const int w = min((int)q.y, N - dx) - max((int)q.x, -dx), h = min((int)q.w, N - dy) - max((int)q.z, -dy);
            c[k] += w > 0 && h > 0 ? (uint32_t)w * (uint32_t)h : 0u;
        }
    }
    bool same = true;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        same = same && __reduce_add_sync(0xffffffffu, c[k]) == __ldg(gn + (k & 2 ? 2 * S * K : 0) + (k & 1 ? 2 * S : 0));
    return same && pcl::rect_corr::ranges_in_raster(r, n, hb, halo_words(N, S), S, lane);
}

// The clips' verdicts (rect_corr.cuh), a warp per clip: the representatives' against
// their window rasters, then the members' against their halo rasters
constexpr int kRectWarps = 4;

__global__ void __launch_bounds__(32 * kRectWarps) halo_verdict_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B,
                                                                      const uint64_t *__restrict__ hbits,
                                                                      const uint32_t *__restrict__ norms, uint64_t n,
                                                                      const unsigned long long *d_n, pcl_record *out) {
    namespace rc = pcl::rect_corr;
    const uint64_t clips = (uint64_t)A.n_clips + B.n_clips;
    if (d_n && *d_n < n) n = *d_n;
    if (!rc::verdicts_pay(n, clips)) return;
    __shared__ short4 ranges[kRectWarps][rc::kRectMax];
    const Geo g = make_geo(prm);
    const int N = g.N, S = g.S, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int psh = (g.p & (g.p - 1)) == 0 ? 31 - __clz(g.p) : -1;
    short4 *r = ranges[warp];
    for (uint64_t k = (uint64_t)blockIdx.x * kRectWarps + warp; k < clips; k += (uint64_t)gridDim.x * kRectWarps) {
        bool ok = false;
        if (k < A.n_clips) {
            ok = rc::window_verdict(A, (uint32_t)k, g, psh, r, lane);
        } else {
            const uint32_t c = (uint32_t)(k - A.n_clips), o = __ldg(B.rect_off + c);
            const int m = (int)(__ldg(B.rect_off + c + 1) - o);
            if (m >= 0 && m <= rc::kRectMax) {
                __syncwarp();  // the previous clip's ranges are no longer read
                rc::stage_rects(reinterpret_cast<const int4 *>(B.rects) + o, m, g.p, psh, -S, N + S, r, lane);
                __syncwarp();
                ok = ranges_are_halo(r, m, hbits + (size_t)c * halo_side(N, S) * halo_words(N, S),
                                     norms + (size_t)c * norms_stride(N, S), g, lane);
            }
        }
        if (lane == 0) *rc::verdict_at(out, k) = ok ? 1 : 0;
    }
}

// One warp per pair: the record from the rectangles (rect_corr.cuh; A's cut to
// its window, B's to the halo) for clips of few enough rectangles that share no
// pixel and are the rasters (the buffers may have been written again, and b may be
// another set of clips than the halo rasters were made from), every shift's
// overlap against the tabulated n_B(s).  The other pairs
// get a record with flags = kRectPending, for halo_pair_kernel.  A pair decided
// here counts as one group of shifts in stats.
__global__ void __launch_bounds__(32 * kRectWarps, 8) halo_rect_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B,
                                                                    const uint64_t *__restrict__ hbits,
                                                                    const uint32_t *__restrict__ norms,
                                                                    const pcl_pair *pairs, uint64_t npairs,
                                                                    const unsigned long long *d_n, pcl_record *out,
                                                                    unsigned long long *stats, bool verdicts) {
    namespace rc = pcl::rect_corr;
    if (d_n && *d_n < npairs) npairs = *d_n;
    verdicts = verdicts && rc::verdicts_pay(npairs, (uint64_t)A.n_clips + B.n_clips);
    extern __shared__ __align__(16) unsigned char smem[];
    const Geo g = make_geo(prm);
    const int N = g.N, S = g.S, K = 2 * S + 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int psh = (g.p & (g.p - 1)) == 0 ? 31 - __clz(g.p) : -1;
    const rc::Scratch s = rc::scratch_at(smem + warp * rc::scratch_bytes(S), S);
    const uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const bool rects = rc::has_rects(A) && rc::has_rects(B);
    unsigned long long done_here = 0;
    for (uint64_t t = w0; t < npairs; t += nw) {  // warp-uniform
        const pcl_pair pr = pairs[t];
        pcl_record rec{};
        rec.a = pr.a;
        rec.b = pr.b;
        rec.mode = PCL_MODE_COSINE;
        if (pr.a >= A.n_clips || pr.b >= B.n_clips) {
            rec.flags = PCL_GATE_BAD_INDEX;
            if (lane == 0) out[t] = rec;
            continue;
        }
        const uint64_t pa = A.pop[pr.a];
        const uint32_t oa = rects ? __ldg(A.rect_off + pr.a) : 0u, ob = rects ? __ldg(B.rect_off + pr.b) : 0u;
        const int na = rects ? (int)(__ldg(A.rect_off + pr.a + 1) - oa) : 0;
        const int nb = rects ? (int)(__ldg(B.rect_off + pr.b + 1) - ob) : 0;
        bool ok = rects && pa != 0 && na >= 0 && nb >= 0 && na <= rc::kRectMax && nb <= rc::kRectMax;
        if (verdicts) ok = ok && out[t].reserved != 0;
        if (ok) {
            __syncwarp();  // the scratch's previous contents are no longer read
            const uint32_t aa = rc::stage_rects(reinterpret_cast<const int4 *>(A.rects) + oa, na, g.p, psh, 0, N, s.ra, lane);
            rc::stage_rects(reinterpret_cast<const int4 *>(B.rects) + ob, nb, g.p, psh, -S, N + S, s.rb, lane);
            __syncwarp();
            ok = verdicts || (rc::ranges_are_raster(s.ra, na, aa, A, pr.a, g, lane) &&
                              ranges_are_halo(s.rb, nb, hbits + (size_t)pr.b * halo_side(N, S) * halo_words(N, S),
                                              norms + (size_t)pr.b * norms_stride(N, S), g, lane));
        }
        if (!ok) {
            rec.flags = rc::kRectPending;
            if (lane == 0) out[t] = rec;
            continue;
        }
        const uint32_t *gn = norms + (size_t)pr.b * norms_stride(N, S);
        Best best{0, 0, 0, 0, false};
        rc::rect_surface(s, na, nb, S, lane, [&](uint32_t c, int dx, int dy) {
            const Best cand{c, __ldg(gn + (dy + S) * K + dx + S), dx, dy, true};
            if (before(cand, best, pa)) best = cand;
        });
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const Best other{__shfl_xor_sync(0xffffffffu, best.c, o), __shfl_xor_sync(0xffffffffu, best.n, o),
                             __shfl_xor_sync(0xffffffffu, best.dx, o), __shfl_xor_sync(0xffffffffu, best.dy, o),
                             __shfl_xor_sync(0xffffffffu, (int)best.valid, o) != 0};
            if (before(other, best, pa)) best = other;
        }
        if (lane == 0) out[t] = halo_record(prm, g, pr, pa, best);
        ++done_here;
    }
    if (lane == 0 && stats && done_here) {
        atomicAdd(stats + 2, done_here);
        atomicAdd(stats + 3, done_here * (unsigned long long)(K * (2 * S / 8 + 1)));
    }
}

// One CTA per pending pair: CTA b of a grid of G owns the pairs b, b + G, .. and
// looks at kThreads of them at a time (as in the exact scan: neighbours in a list are
// pending together; 1,000 pairs of clips of 100 rectangles of 256x256 px 0.16 ms, with
// consecutive pairs per CTA 7.2)
template <int NW>
__global__ void __launch_bounds__(kThreads, NW >= 8 ? 2 : 4) halo_pair_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B,
                                                             const uint64_t *__restrict__ hbits,
                                                             const uint32_t *__restrict__ norms, const pcl_pair *pairs,
                                                             uint64_t npairs, const unsigned long long *d_n,
                                                             pcl_record *out, unsigned long long *stats) {
    constexpr int N = 64 * NW;
    const Geo g = make_geo(prm);
    const int S = g.S, NH = halo_side(N, S), NWH = halo_words(N, S), K = 2 * S + 1, KK = K * K;
    const int RW = NWH + 1;  // halo row words read: NWH and one zero word of padding
    const int SA = a_stride(NW), SH = h_stride(NWH);  // row strides in shared memory
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sa = reinterpret_cast<uint64_t *>(smem);          // [N][SA]
    uint64_t *sh = sa + (size_t)N * SA;                         // [NH][SH]
    uint32_t *sn = reinterpret_cast<uint32_t *>(sh + (size_t)NH * SH);  // [K*K]
    Best *wb = reinterpret_cast<Best *>(sn + ((KK + 3) & ~3));  // [warps]
    uint32_t *order = reinterpret_cast<uint32_t *>(wb + kThreads / 32);  // [1024] tasks, best first
    uint32_t *hist = order + 1024;                              // [256]
    unsigned long long *bestcn = reinterpret_cast<unsigned long long *>(hist + pcl::exact_dev::kBuckets);  // best (c << 32 | n) so far
    uint32_t *hbd = reinterpret_cast<uint32_t *>(bestcn + 1);   // [2 NH]: hrow, hcol of B
    uint32_t *rhb = hbd + 2 * NH, *chb = rhb + K;               // [K] Rh(dy), [K] Ch(dx)
    uint32_t *ntasks_done = chb + K, *maxkey = ntasks_done + 1;  // [1] each
    uint16_t *prA = reinterpret_cast<uint16_t *>(ntasks_done + 2);  // [2N]: A's row, column counts
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    // row starts of A's window and of the halo raster, and each warp's segments
    // of equal row pairs (the exact scan's: exact_dev.cuh)
    uint32_t *starts = reinterpret_cast<uint32_t *>(prA + 2 * N), *starts_h = starts + N / 32;
    uint16_t *seg = reinterpret_cast<uint16_t *>(starts_h + (NH + 31) / 32) + warp * (2 * N + 2), *len = seg + N + 1;
    if (d_n && *d_n < npairs) npairs = *d_n;
    __shared__ uint16_t open_s[kThreads];
    __shared__ int count;
    for (uint64_t t0 = blockIdx.x; t0 < npairs; t0 += (uint64_t)gridDim.x * kThreads) {
      __syncthreads();  // the previous list is no longer read
      if (threadIdx.x == 0) count = 0;
      __syncthreads();
      const uint64_t own = t0 + (uint64_t)threadIdx.x * gridDim.x;
      if (own < npairs && out[own].flags == pcl::rect_corr::kRectPending)
          open_s[atomicAdd(&count, 1)] = (uint16_t)threadIdx.x;
      __syncthreads();
      const int n_open = count;
      for (int k_open = 0; k_open < n_open; ++k_open) {
        const uint64_t pid = t0 + (uint64_t)open_s[k_open] * gridDim.x;
        const pcl_pair pr = pairs[pid];
        __syncthreads();  // the previous pair's buffers are no longer read
        const uint64_t *ga = A.bits + (size_t)pr.a * N * NW;
        const uint64_t *gh = hbits + (size_t)pr.b * NH * NWH;
        for (int t = threadIdx.x; t < N * NW; t += blockDim.x) sa[(t / NW) * SA + t % NW] = __ldg(ga + t);
        for (int t = threadIdx.x; t < NH * RW; t += blockDim.x) {
            const int row = t / RW, k = t % RW;
            sh[row * SH + k] = k < NWH ? __ldg(gh + (size_t)row * NWH + k) : 0ull;
        }
        const uint32_t *gn = norms + (size_t)pr.b * norms_stride(N, S);
        for (int t = threadIdx.x; t < KK; t += blockDim.x) sn[t] = __ldg(gn + t);
        for (int t = threadIdx.x; t < 2 * NH; t += blockDim.x) hbd[t] = __ldg(gn + KK + t);
        for (int t = threadIdx.x; t < 2 * N; t += blockDim.x) prA[t] = __ldg(A.prof + (size_t)pr.a * 2 * N + t);
        for (int t = threadIdx.x; t < pcl::exact_dev::kBuckets; t += blockDim.x) hist[t] = 0u;
        if (threadIdx.x == 0) {
            *maxkey = 0u;
            *bestcn = 0ull;
            *ntasks_done = 0u;
        }
        __syncthreads();
        row_starts64(sa, N, NW, SA, starts);
        row_starts64(sh, NH, NWH, SH, starts_h);
        const uint64_t pa = A.pop[pr.a];
        // Upper bounds of c(s): A's row y meets halo row y - dy + S in at most
        // min(r_A(y), hrow) ones, so c(dx, dy) <= Rh(dy) = sum_y min(r_A(y),
        // hrow(y - dy + S)), and c(dx, dy) <= Ch(dx) over the columns; with the
        // moved-window count n_B(s), sim(s) <= min(Rh, Ch) / sqrt(|A| n_B(s)).
        for (int v = warp; v < 2 * K; v += nwarps) {
            const bool col = v >= K;
            const int d = (col ? v - K : v) - S;
            const uint16_t *pa_ = prA + (col ? N : 0);
            const uint32_t *hb_ = hbd + (col ? NH : 0);
            uint32_t sum = 0;
            for (int y = lane; y < N; y += 32) sum += min((uint32_t)pa_[y], hb_[y - d + S]);
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (lane == 0) (col ? chb : rhb)[d + S] = sum;
        }
        __syncthreads();
        Best best{0, 0, 0, 0, false};
        // warp task: (dy, 8 consecutive sd = S - dx starting at a multiple of
        // 8); lanes take rows y and count the 8 shifts from registers as
        // 32-bit words: A's word w lines up with halo bits [32 w + sd, +32),
        // which start in halo word w + sd / 32, the same word for the 8
        // shifts of a task
        const int nch = (2 * S) / 8 + 1, ntask = K * nch;
        // a task can be skipped when every shift's bound is below the best
        // similarity found so far, (cb, nb): U^2 nb < cb^2 n_B(s), exactly in
        // integers (U^2 n < 2^54 up to 512^2); not for an empty A (sim 1
        // for an empty window)
        auto prunable = [&](int task, uint32_t cb, uint32_t nb) -> bool {
            if (pa == 0 || cb == 0) return false;
            const int dy = task / nch - S, sd0 = (task % nch) * 8;
            for (int u = 0; u < 8; ++u) {
                const int sd = sd0 + u;
                if (sd > 2 * S) break;
                const int dx = S - sd;
                const uint32_t n = sn[(dy + S) * K + dx + S];
                if (n == 0) continue;  // c = 0 there: sim 0 < the best
                const uint64_t U = min(rhb[dy + S], chb[dx + S]);
                if (U * U * nb >= (uint64_t)cb * cb * n) return false;
            }
            return true;
        };
        auto eval_task = [&](int task) {
            const int dy = task / nch - S, sd0 = (task % nch) * 8;
            const int qq = sd0 >> 5, rb = sd0 & 31;  // sd = 32 qq + rb + u, rb + u <= 31
            uint32_t cnt[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) cnt[u] = 0;
            const int n = pcl::exact_dev::row_segments<N>(starts, starts_h, NH, S - dy, 0, N, prA, hbd, seg, len, lane);
            for (int i = lane; i < n; i += 32) {
                const int y = seg[i];
                const uint32_t times = len[i];
                // A's row and the halo row into registers once (RW = NW + 2
                // words for 1 <= S <= 32, NW + 1 for S = 0)
                const uint64_t *ra = sa + (size_t)y * SA;
                const uint64_t *rh = sh + (size_t)(y - dy + S) * SH;
                uint32_t a[2 * NW], h[2 * NW + 4];
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const uint64_t v = ra[w];
                    a[2 * w] = (uint32_t)v;
                    a[2 * w + 1] = (uint32_t)(v >> 32);
                }
#pragma unroll
                for (int k = 0; k < NW + 2; ++k) {
                    const uint64_t v = k < RW ? rh[k] : 0ull;
                    h[2 * k] = (uint32_t)v;
                    h[2 * k + 1] = (uint32_t)(v >> 32);
                }
                if (qq == 0) halo_row_counts<2 * NW, 0>(a, h, rb, times, cnt);
                else if (qq == 1) halo_row_counts<2 * NW, 1>(a, h, rb, times, cnt);
                else halo_row_counts<2 * NW, 2>(a, h, rb, times, cnt);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int sd = sd0 + u, dx = S - sd;
                const uint32_t c = __reduce_add_sync(0xffffffffu, cnt[u]);
                if (sd <= 2 * S) {
                    const Best cand{c, sn[(dy + S) * K + dx + S], dx, dy, true};
                    if (before(cand, best, pa)) best = cand;
                }
            }
        };
        // best first: tasks in buckets of their largest bound of U^2 / n_B (floats,
        // descending); they only order the work, the skip test above is exact
        auto task_key = [&](int t) -> float {
            const int dy = t / nch - S, sd0 = (t % nch) * 8;
            float kb = 0.0f;
            for (int u = 0; u < 8 && sd0 + u <= 2 * S; ++u) {
                const int dx = S - (sd0 + u);
                const uint32_t n = sn[(dy + S) * K + dx + S];
                const float U = (float)min(rhb[dy + S], chb[dx + S]);
                if (n) kb = fmaxf(kb, U * U / (float)n);
            }
            return kb;
        };
        {
            constexpr int PER = (65 * 9 + kThreads - 1) / kThreads;  // S <= 32: at most 65 x 9 tasks
            float kb[PER], top = 0.0f;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int t = threadIdx.x + k * kThreads;
                kb[k] = t < ntask ? task_key(t) : 0.0f;
                top = fmaxf(top, kb[k]);
            }
            const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(top));  // not negative: ordered as integers
            if (lane == 0) atomicMax(maxkey, m);
            __syncthreads();
            pcl::exact_dev::bucket_order<PER>(
                ntask, __uint_as_float(*maxkey), hist, [&](int, int k) { return kb[k]; },
                [&](int t) { return (uint32_t)t; }, order);
        }
        // warp w takes positions w, w + nwarps, ..: each lane tests one of its
        // next 32, the first that is left is counted, and the rest tested again
        // against the best known then
        for (int q0 = warp; q0 < ntask; q0 += 32 * nwarps) {
            const int q = q0 + lane * nwarps;
            const int task_l = q < ntask ? (int)order[q] : 0;
            bool open = q < ntask;
            for (;;) {
                const unsigned long long bc =
                    __shfl_sync(0xffffffffu, *reinterpret_cast<volatile unsigned long long *>(bestcn), 0);
                open = open && !prunable(task_l, (uint32_t)(bc >> 32), (uint32_t)bc);
                const unsigned m = __ballot_sync(0xffffffffu, open);
                if (!m) break;
                const int src = __ffs(m) - 1;
                if (lane == src) open = false;
                eval_task(__shfl_sync(0xffffffffu, task_l, src));
                if (lane == 0) {
                    atomicAdd(ntasks_done, 1u);
                    if (best.valid && best.c > 0 && best.n > 0) {  // raise the shared best to this warp's
                        unsigned long long old = *reinterpret_cast<volatile unsigned long long *>(bestcn), seen;
                        do {
                            seen = old;
                            const uint32_t c0 = (uint32_t)(seen >> 32), n0 = (uint32_t)seen;
                            if (c0 && (uint64_t)best.c * best.c * n0 <= (uint64_t)c0 * c0 * best.n) break;
                            old = atomicCAS(bestcn, seen, ((unsigned long long)best.c << 32) | best.n);
                        } while (old != seen);
                    }
                }
            }
        }
        if (lane == 0) wb[warp] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            if (stats) {
                atomicAdd(stats + 2, (unsigned long long)*ntasks_done);
                atomicAdd(stats + 3, (unsigned long long)ntask);
            }
            Best b = wb[0];
            for (int w = 1; w < nwarps; ++w)
                if (before(wb[w], b, pa)) b = wb[w];
            out[pid] = halo_record(prm, g, pr, pa, b);
        }
      }
    }
}

size_t raster_smem(const Geo &g) {
    const int NH = halo_side(g.N, g.S), NWH = halo_words(g.N, g.S), K = 2 * g.S + 1;
    return 4ull * NH * row_stride(NWH) + 4ull * K * K + 2ull * K * cnt_stride(NH);
}

size_t pair_smem(const Geo &g) {
    const int NH = halo_side(g.N, g.S), NWH = halo_words(g.N, g.S), K = 2 * g.S + 1;
    return 8ull * g.N * a_stride(g.nw) + 8ull * NH * h_stride(NWH) + 4ull * (((size_t)K * K + 3) & ~size_t(3)) +
           sizeof(Best) * (kThreads / 32) + 4ull * (1024 + pcl::exact_dev::kBuckets) + 8 + 4ull * (2 * NH + 2 * K + 2) + 2ull * 2 * g.N +
           4ull * (g.N / 32 + (NH + 31) / 32) + (kThreads / 32) * 2ull * (2 * g.N + 2) + 16;
}

template <int NW>
cudaError_t launch_pair(const pcl_params &prm, const Geo &g, const pcl_clipset &a, const pcl_clipset &b,
                        const uint64_t *hb, const uint32_t *nb, const pcl_pair *pairs, uint64_t n,
                        const unsigned long long *d_n, pcl_record *out, int num_sms, unsigned long long *stats,
                        cudaStream_t st) {
    const size_t sm = pair_smem(g);
    cudaError_t e = cudaFuncSetAttribute(halo_pair_kernel<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, halo_pair_kernel<NW>, kThreads, sm);
    if (e != cudaSuccess) return e;
    const uint64_t cap = (uint64_t)num_sms * (uint64_t)(per_sm > 0 ? per_sm : 1);
    {
        const size_t rs = kRectWarps * pcl::rect_corr::scratch_bytes(g.S);
        e = cudaFuncSetAttribute(halo_rect_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rs);
        int rect_sm = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&rect_sm, halo_rect_kernel, 32 * kRectWarps, rs);
        if (e != cudaSuccess) return e;
        const uint64_t most = (uint64_t)num_sms * (uint64_t)(rect_sm > 0 ? rect_sm : 1);
        const uint64_t need = (n + kRectWarps - 1) / kRectWarps;
        namespace rc = pcl::rect_corr;
        const uint64_t clips = (uint64_t)a.n_clips + b.n_clips, grid = (clips + kRectWarps - 1) / kRectWarps;
        const bool verdicts = clips && rc::has_rects(a) && rc::has_rects(b) && rc::verdicts_pay(n, clips);
        if (verdicts) {
            const uint64_t full = (uint64_t)num_sms * 16, blocks = (n + 255) / 256;
            halo_verdict_kernel<<<(unsigned)(grid < full ? grid : full), 32 * kRectWarps, 0, st>>>(prm, a, b, hb, nb, n,
                                                                                                  d_n, out);
            rc::pair_verdict_kernel<<<(unsigned)(blocks < full ? blocks : full), 256, 0, st>>>(
                a.n_clips, b.n_clips, a.n_clips, clips, pairs, n, d_n, out);
        }
        halo_rect_kernel<<<(unsigned)(need < most ? need : most), 32 * kRectWarps, rs, st>>>(
            prm, a, b, hb, nb, pairs, n, d_n, out, stats, verdicts);
    }
    halo_pair_kernel<NW><<<(unsigned)(n < cap ? n : cap), kThreads, sm, st>>>(prm, a, b, hb, nb, pairs, n, d_n, out,
                                                                             stats);
    return cudaGetLastError();
}

pcl_status fail(pcl_ctx *ctx, pcl_status s, const char *m) {
    ctx->err = m;
    return s;
}

pcl_status cuda_fail(pcl_ctx *ctx, cudaError_t e, const char *where) {
    ctx->err = std::string(where) + ": " + cudaGetErrorString(e);
    return PCL_ERR_CUDA;
}

bool halo_geometry_ok(const Geo &g) { return g.S <= 32 && g.S <= g.N / 2; }

}  // namespace

extern "C" {

pcl_status pcl_halo_sizes_get(const pcl_params *P, uint32_t n_clips, uint64_t *hbits_bytes, uint64_t *norms_bytes) {
    if (pcl_params_validate(P) != PCL_OK || !hbits_bytes || !norms_bytes) return PCL_ERR_INVALID;
    const Geo g = make_geo(*P);
    if (!halo_geometry_ok(g)) return PCL_ERR_UNSUPPORTED;
    *hbits_bytes = 8ull * n_clips * halo_side(g.N, g.S) * halo_words(g.N, g.S);
    *norms_bytes = 4ull * n_clips * (uint64_t)norms_stride(g.N, g.S);
    return PCL_OK;
}

pcl_status pcl_rasterize_halo(pcl_ctx *ctx, const pcl_params *P, const pcl_clipset *cs, uint64_t *d_hbits,
                              uint32_t *d_norms, pcl_stream stream) {
    if (!ctx) return PCL_ERR_INVALID;
    ctx->err.clear();
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaSetDevice");
    if (pcl_params_validate(P) != PCL_OK) return fail(ctx, PCL_ERR_INVALID, "pcl_rasterize_halo: invalid parameters");
    const Geo g = make_geo(*P);
    if (!halo_geometry_ok(g)) return fail(ctx, PCL_ERR_UNSUPPORTED, "pcl_rasterize_halo: needs S <= 32 and S <= N/2");
    if (!cs || (cs->n_clips && (!cs->rect_off || !cs->rects || !d_hbits || !d_norms)))
        return fail(ctx, PCL_ERR_INVALID, "pcl_rasterize_halo: NULL buffer");
    if (cs->n_clips == 0) return PCL_OK;
    const size_t sm = raster_smem(g);
    e = cudaFuncSetAttribute(halo_raster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess) {
        halo_raster_kernel<<<cs->n_clips, kRasterThreads, sm, (cudaStream_t)stream>>>(*P, *cs, d_hbits, d_norms);
        e = cudaGetLastError();
    }
    return e == cudaSuccess ? PCL_OK : cuda_fail(ctx, e, "halo raster kernel");
}

pcl_status pcl_match_halo(pcl_ctx *ctx, const pcl_params *P, const pcl_clipset *a, const pcl_clipset *b,
                          const uint64_t *d_hbits_b, const uint32_t *d_norms_b, const pcl_pair *d_pairs, uint64_t n,
                          const uint64_t *d_n, pcl_record *d_out, pcl_stream stream) {
    if (!ctx) return PCL_ERR_INVALID;
    ctx->err.clear();
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaSetDevice");
    if (pcl_params_validate(P) != PCL_OK) return fail(ctx, PCL_ERR_INVALID, "pcl_match_halo: invalid parameters");
    const Geo g = make_geo(*P);
    if (!halo_geometry_ok(g)) return fail(ctx, PCL_ERR_UNSUPPORTED, "pcl_match_halo: needs S <= 32 and S <= N/2");
    if (!a || !b || (n && (!d_pairs || !d_out || !d_hbits_b || !d_norms_b)) ||
        (a->n_clips && (!a->bits || !a->pop || !a->prof)))
        return fail(ctx, PCL_ERR_INVALID, "pcl_match_halo: NULL buffer");
    if (n == 0) return PCL_OK;
    const auto *dn = reinterpret_cast<const unsigned long long *>(d_n);
    cudaStream_t st = (cudaStream_t)stream;
    switch (g.nw) {
        case 1: e = launch_pair<1>(*P, g, *a, *b, d_hbits_b, d_norms_b, d_pairs, n, dn, d_out, ctx->num_sms,
                                       ctx->d_stats, st); break;
        case 2: e = launch_pair<2>(*P, g, *a, *b, d_hbits_b, d_norms_b, d_pairs, n, dn, d_out, ctx->num_sms,
                                       ctx->d_stats, st); break;
        case 4: e = launch_pair<4>(*P, g, *a, *b, d_hbits_b, d_norms_b, d_pairs, n, dn, d_out, ctx->num_sms,
                                       ctx->d_stats, st); break;
        case 8: e = launch_pair<8>(*P, g, *a, *b, d_hbits_b, d_norms_b, d_pairs, n, dn, d_out, ctx->num_sms,
                                       ctx->d_stats, st); break;
        default: return fail(ctx, PCL_ERR_UNSUPPORTED, "pcl_match_halo: raster side");
    }
    return e == cudaSuccess ? PCL_OK : cuda_fail(ctx, e, "halo pair kernel");
}

}  // extern "C"
