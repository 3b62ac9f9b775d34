// Device code of the exact window scan (Sec. 2.2.1, Eq. 2: c(s) for the
// shifts of the marker window by popcount, the best shift by the exact argmax
// with the tie order), shared by the exact pair kernel (fft.cu) and the
// mixed-batch kernel: the path of 512^2 rasters and the exact-scan engine.
#pragma once

#include "gates.cuh"

namespace pcl {
namespace exact_dev {

// Exact window scan (N = 64 NW: 512^2, where the FFT body's buffers exceed
// shared memory, and 128^2 / 256^2 as the exact-scan engine): c(s) = sum_x
// A(x) B(x - s) counted with AND + popcount for the shifts |dx|, |dy| <= S
// (S <= SMAX <= 32) that the profile bounds do not exclude -- the definition
// itself, so the record is the oracle's.  Both rasters are staged in shared memory (2 N²/8 bytes).  Warps
// take (dy, 8 consecutive dx starting at a multiple of 8); lanes take row pairs
// (A row y, B row y - dy) as 32-bit words and count the 8 shifts of a row pair
// from registers, one funnel shift per word and shift: B's row moved by
// dx = 32 q + r is word w - q funnel-shifted by r with word w - q - 1, and q is
// the same for the 8 shifts of a task because the chunk starts at a multiple
// of 8.  No phase-correlation surface is formed (pcm fields 0).  The caller has
// checked the indices, emptiness and gates.
// Only different row pairs are counted: a raster of rectangles has runs of
// equal rows (at 512^2 about 45 of them per clip), so for one dy the pairs
// (A row y, B row y - dy) fall into segments of equal pairs, at most one per run
// of either clip; a segment is counted once, times its length, and segments
// where either row is empty are left out.  12,001 same-seed pairs of 512^2 px:
// 5.3 ms against 24.9-26.4 counting every row.

// bit y % 32 of word y / 32: row y of the N staged rows differs from row y - 1
// (row 0: set); rows of NV 16-byte vectors at stride SV
__device__ __forceinline__ void row_starts(const uint4 *rows, int n_rows, int NV, int SV, uint32_t *starts) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int w = warp; w < (n_rows + 31) / 32; w += nwarps) {
        const int y = 32 * w + lane;
        bool diff = y == 0;
        if (y > 0 && y < n_rows)
            for (int v = 0; v < NV && !diff; ++v) {
                const uint4 a = rows[y * SV + v], b = rows[(y - 1) * SV + v];
                diff = ((a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w)) != 0u;
            }
        const uint32_t m = __ballot_sync(0xffffffffu, diff);
        if (lane == 0) starts[w] = m;
    }
}

// The segments of equal row pairs (A row j, B row j + off), j in [j0, j1), whose
// rows both hold ones: first rows in seg[0 .. count), lengths in len[..]; seg
// has N + 1 entries.  sa, sb: row starts (row_starts; sb of nb rows); count_a,
// count_b: ones per row.  One warp; the result is warp-uniform.
template <int N, typename CA, typename CB>
__device__ __forceinline__ int row_segments(const uint32_t *sa, const uint32_t *sb, int nb, int off, int j0, int j1,
                                            const CA *count_a, const CB *count_b, uint16_t *seg, uint16_t *len,
                                            int lane) {
    constexpr int K = N / 32;  // rows per lane
    static_assert(K <= 16, "a lane's rows fit a word");
    const int y = K * lane;
    uint32_t m = sa[y >> 5] >> (y & 31);
    const int b = y + off, wi = b >= 0 ? b >> 5 : -((31 - b) >> 5), nw = (nb + 31) >> 5;
    const uint32_t lo = wi >= 0 && wi < nw ? sb[wi] : 0u, hi = wi + 1 >= 0 && wi + 1 < nw ? sb[wi + 1] : 0u;
    m |= __funnelshift_r(lo, hi, b & 31);
    // rows [j0, j1) only; j0 starts a segment
    const int l = j0 - y, h = j1 - y;
    if (l >= 0 && l < K) m |= 1u << l;
    m &= l <= 0 ? 0xffffffffu : l >= 32 ? 0u : 0xffffffffu << l;
    m &= h >= 32 ? 0xffffffffu : h <= 0 ? 0u : (1u << h) - 1u;
    m &= (1u << K) - 1u;
    const int n = __popc(m);
    int x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    const int total = __shfl_sync(0xffffffffu, x, 31);
    __syncwarp();  // the previous task's segments are no longer read
    for (int at = x - n; m; ++at, m &= m - 1u) seg[at] = (uint16_t)(y + __ffs(m) - 1);
    if (lane == 0) seg[total] = (uint16_t)j1;
    __syncwarp();
    int kept = 0;
    for (int i0 = 0; i0 < total; i0 += 32) {  // in place: kept <= i0
        const int i = i0 + lane;
        const int s = i < total ? seg[i] : 0, e = i < total ? seg[i + 1] : 0;
        const bool keep = i < total && count_a[s] != 0 && count_b[s + off] != 0;
        const unsigned k = __ballot_sync(0xffffffffu, keep);  // also orders the reads before the writes
        const int at = kept + __popc(k & ((1u << lane) - 1u));
        if (keep) {
            seg[at] = (uint16_t)s;
            len[at] = (uint16_t)(e - s);
        }
        kept += __popc(k);
        __syncwarp();
    }
    return kept;
}

template <int NW32, int Q>
__device__ __forceinline__ void exact_row_counts(const uint32_t (&a)[NW32], const uint32_t (&bp)[NW32 + 3], int rb,
                                                 uint32_t times, uint32_t (&cnt)[8]) {
    // bp[i] = B's word i - 2 (zero outside the row); B moved by 32 Q + r has
    // word w = funnel(b[w - Q - 1], b[w - Q], r) = funnel(bp[w + 1 - Q], bp[w + 2 - Q], r)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int r = rb + u;  // 0..31
        uint32_t x[NW32];
#pragma unroll
        for (int w = 0; w < NW32; ++w) x[w] = a[w] & __funnelshift_l(bp[w + 1 - Q], bp[w + 2 - Q], r);
        cnt[u] += times * popc_sum<NW32>(x);
    }
}

// Order of the ntask tasks by bound, largest bucket first, into order[]: a
// counting sort into 256 buckets of equal width (hist: 256 u32 of shared memory,
// zeroed).  bound(t, k) is task t's bound as a float (the thread's k-th task), top at least the largest;
// order[] gets key(t).  Inside a bucket the order is arbitrary.  (A bitonic
// sort took 36 to 55 barriers, this takes three.)  Returns with a barrier.
constexpr int kBuckets = 256;
__device__ __forceinline__ int bucket_of(float bound, float top) {
    return top > 0.0f ? min(kBuckets - 1, (int)((top - bound) * ((float)kBuckets / top))) : 0;
}
template <int MAXT, typename Bound, typename Key, typename Out>
__device__ __forceinline__ void bucket_order(int ntask, float top, uint32_t *hist, Bound bound, Key key, Out *order) {
    const int lane = threadIdx.x & 31;
    int bk[MAXT], rank[MAXT];
#pragma unroll
    for (int k = 0; k < MAXT; ++k) {
        const int t = threadIdx.x + k * blockDim.x;
        if (t < ntask) {
            bk[k] = bucket_of(bound(t, k), top);
            rank[k] = (int)atomicAdd(hist + bk[k], 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // exclusive scan, eight buckets a lane
        constexpr int R = kBuckets / 32;
        uint32_t v[R], sum = 0;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            v[k] = sum;
            sum += hist[R * lane + k];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
#pragma unroll
        for (int k = 0; k < R; ++k) hist[R * lane + k] = x - sum + v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < MAXT; ++k) {
        const int t = threadIdx.x + k * blockDim.x;
        if (t < ntask) order[hist[bk[k]] + rank[k]] = key(t);
    }
    __syncthreads();
}

// threads of a CTA that runs exact_body: at 512^2 two CTAs of ten warps fill
// the SM's shared memory, at the smaller sizes CTAs of four warps leave room
// for six and more, and their barriers cost less
template <int NW>
constexpr int exact_threads() {
    return NW == 8 ? 320 : 128;
}

template <int NW, int SMAX>
__device__ __forceinline__ void exact_body(const pcl_params &prm, const pcl_clipset &A, const pcl_clipset &B,
                                           const pcl_pair pr, pcl_record *dst,
                                           unsigned long long *stats = nullptr) {
    static_assert(SMAX <= 32 && NW >= 2, "shift words: q in {-1, 0, 1}; rows of whole 16-byte vectors");
    constexpr int N = 64 * NW, NW32 = 2 * NW, NV = NW32 / 4;  // 32-bit words and 16-byte vectors per row
    // row stride in shared memory: an odd number of vectors, so that the 8
    // lanes of a quarter-warp reading 8 consecutive rows hit 8 bank groups
    constexpr int SV = NV | 1;
    const Geo g = make_geo(prm);
    const int S = g.S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    extern __shared__ __align__(16) unsigned char smem[];
    uint4 *sa = reinterpret_cast<uint4 *>(smem);
    uint4 *sb = sa + N * SV;
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(sb + N * SV);  // [32]
    uint32_t *rbound = reinterpret_cast<uint32_t *>(keys + 32);                      // [2 SMAX + 1]: R(dy)
    uint32_t *cbound = rbound + 2 * SMAX + 1;                                         // [2 SMAX + 1]: C(dx)
    uint32_t *lbest = cbound + 2 * SMAX + 1;  // [0]: L, [1]: tasks evaluated
    constexpr int MAXTASK = (2 * SMAX + 1) * (2 * ((SMAX + 7) / 8) + 1);             // tasks at S = SMAX
    uint32_t *order = lbest + 4;                                                      // [MAXTASK] keys in order
    uint32_t *hist = order + MAXTASK;                                                 // [256]
    uint16_t *prof = reinterpret_cast<uint16_t *>(hist + kBuckets + (MAXTASK & 1));   // [2][2N]: A's, B's
    uint32_t *starts = reinterpret_cast<uint32_t *>(prof + 4 * N);                    // [2][N / 32]: A's, B's row starts
    uint16_t *seg = reinterpret_cast<uint16_t *>(starts + 2 * (N / 32)) + warp * (2 * N + 2), *len = seg + N + 1;
    const uint4 *ga = reinterpret_cast<const uint4 *>(A.bits + (size_t)pr.a * N * NW);
    const uint4 *gb = reinterpret_cast<const uint4 *>(B.bits + (size_t)pr.b * N * NW);
    __syncthreads();  // the shared memory may still be read by the previous item
    for (int t = threadIdx.x; t < N * NV; t += blockDim.x) {
        const int st = (t / NV) * SV + t % NV;
        sa[st] = __ldg(ga + t);
        sb[st] = __ldg(gb + t);
    }
    for (int t = threadIdx.x; t < 2 * N; t += blockDim.x) {
        prof[t] = __ldg(A.prof + (size_t)pr.a * 2 * N + t);
        prof[2 * N + t] = __ldg(B.prof + (size_t)pr.b * 2 * N + t);
    }
    for (int t = threadIdx.x; t < kBuckets; t += blockDim.x) hist[t] = 0u;
    if (threadIdx.x == 0) lbest[0] = lbest[1] = 0u;
    __syncthreads();
    row_starts(sa, N, NV, SV, starts);
    row_starts(sb, N, NV, SV, starts + N / 32);
    const int K = 2 * S + 1;
    // Upper bounds from the projection profiles (the bound of gate G2): rows y
    // of A and y - dy of B overlap in at most min(r_A(y), r_B(y - dy)) pixels,
    // so c(dx, dy) <= R(dy) = sum_y min(r_A(y), r_B(y - dy)), and likewise
    // c(dx, dy) <= C(dx) over the columns.
    for (int v = warp; v < 2 * K; v += nwarps) {
        const bool col = v >= K;
        const int d = (col ? v - K : v) - S;
        const uint16_t *pa_ = prof + (col ? N : 0), *pb_ = prof + 2 * N + (col ? N : 0);
        uint32_t sum = 0;
        for (int y = lane; y < N; y += 32) {
            const int yb = y - d;
            if (yb >= 0 && yb < N) sum += min((uint32_t)pa_[y], (uint32_t)pb_[yb]);
        }
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0) (col ? cbound : rbound)[d + S] = sum;
    }
    __syncthreads();
    // dx chunks [8 c, 8 c + 7] for c = floor(-S / 8) .. floor(S / 8); a task
    // (dy, chunk) is bounded by min(R(dy), max of C over its shifts)
    const int c0 = -((S + 7) / 8), nch = S / 8 - c0 + 1;
    auto task_bound = [&](int task) -> uint32_t {
        const int dy = task / nch - S, dx0 = (c0 + task % nch) * 8;
        uint32_t cm = 0;
        for (int u = 0; u < 8; ++u) {
            const int dx = dx0 + u;
            if (dx >= -S && dx <= S) cm = max(cm, cbound[dx + S]);
        }
        return min(rbound[dy + S], cm);
    };
    unsigned long long best = 0ull;
    // c(s) for the 8 shifts of one task; returns their largest overlap
    auto eval_task = [&](int task) -> uint32_t {
        const int dy = task / nch - S, dx0 = (c0 + task % nch) * 8;  // -32 <= dx0 <= 32
        const int q = (dx0 + 32) / 32 - 1, rb = dx0 - 32 * q;        // dx0 = 32 q + rb, rb in {0, 8, 16, 24}
        uint32_t cnt[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) cnt[u] = 0;
        const int j0 = dy > 0 ? dy : 0, j1 = dy < 0 ? N + dy : N;
        const int n = row_segments<N>(starts, starts + N / 32, N, -dy, j0, j1, prof, prof + 2 * N, seg, len, lane);
        for (int i = lane; i < n; i += 32) {
            const int j = seg[i];
            const uint32_t times = len[i];
            uint32_t a[NW32], bp[NW32 + 3];
            bp[0] = bp[1] = bp[NW32 + 2] = 0u;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const uint4 x = sa[j * SV + v], y = sb[(j - dy) * SV + v];
                a[4 * v] = x.x, a[4 * v + 1] = x.y, a[4 * v + 2] = x.z, a[4 * v + 3] = x.w;
                bp[4 * v + 2] = y.x, bp[4 * v + 3] = y.y, bp[4 * v + 4] = y.z, bp[4 * v + 5] = y.w;
            }
            if (q < 0) exact_row_counts<NW32, -1>(a, bp, rb, times, cnt);
            else if (q == 0) exact_row_counts<NW32, 0>(a, bp, rb, times, cnt);
            else exact_row_counts<NW32, 1>(a, bp, rb, times, cnt);
        }
        uint32_t cmax = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int dx = dx0 + u;
            const uint32_t c = __reduce_add_sync(0xffffffffu, cnt[u]);
            if (dx >= -S && dx <= S) {
                const unsigned long long k = shift_key(c, dx, dy, S);
                best = k > best ? k : best;
                cmax = max(cmax, c);
            }
        }
        return cmax;
    };
    // Best first: the tasks by bound, descending by bucket (keys bound << 12 |
    // task); warp w takes positions w, w + nwarps, ...  The first round (the
    // largest bounds) sets L, the largest overlap counted so far, and every
    // counted task raises it (shared atomic max).  A task whose bound is below L
    // is skipped: it holds no shift whose overlap reaches the best, so the
    // argmax and its ties are the full scan's.  A warp stops at its first
    // position in a bucket that lies below L's: all bounds after it are below L.
    const int ntask = K * nch;  // <= MAXTASK
    float top;
    {
        uint32_t mr = 0, mc = 0;
        for (int k = lane; k < K; k += 32) {
            mr = max(mr, rbound[k]);
            mc = max(mc, cbound[k]);
        }
        top = (float)min(__reduce_max_sync(0xffffffffu, mr), __reduce_max_sync(0xffffffffu, mc));
    }
    constexpr int PER = (MAXTASK + exact_threads<NW>() - 1) / exact_threads<NW>();
    bucket_order<PER>(
        ntask, top, hist, [&](int t, int) { return (float)task_bound(t); },
        [&](int t) { return (task_bound(t) << 12) | (uint32_t)t; }, order);
    for (int p = warp; p < ntask; p += nwarps) {
        const uint32_t key = order[p];
        const uint32_t lnow = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(lbest), 0);
        if ((key >> 12) < lnow) {  // warp-uniform
            if (bucket_of((float)(key >> 12), top) > bucket_of((float)lnow, top)) break;
            continue;
        }
        const uint32_t cm = eval_task((int)(key & 4095u));
        if (lane == 0) {
            atomicMax(lbest, cm);
            atomicAdd(lbest + 1, 1u);
        }
    }
    if (lane == 0) keys[warp] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        if (stats) {
            atomicAdd(stats, (unsigned long long)lbest[1]);
            atomicAdd(stats + 1, (unsigned long long)(K * nch));
        }
        unsigned long long bk = 0ull;
        for (int w = 0; w < nwarps; ++w) bk = keys[w] > bk ? keys[w] : bk;
        const int dx = S - (int)(bk & 0xffu), dy = S - (int)((bk >> 8) & 0xffu);
        const uint32_t cb = (uint32_t)(bk >> 32);
        const uint64_t pa = A.pop[pr.a], pb = B.pop[pr.b];
        pcl_record rec{};
        rec.a = pr.a;
        rec.b = pr.b;
        rec.mode = PCL_MODE_COSINE;
        rec.dx_dbu = dx * g.p;
        rec.dy_dbu = dy * g.p;
        rec.score = cb;
        float sim = (pa && pb) ? (float)cb / sqrtf((float)pa * (float)pb) : 0.0f;
        uint16_t fl = PCL_F_ALIGNED;
        const float T = (float)prm.cos_num / (float)prm.cos_den;
        if (pa && pb && fabsf(sim - T) < prm.near_band) {
            fl |= PCL_F_NEAR_BAND;
            sim = (float)((double)cb / sqrt((double)pa * (double)pb));
        }
        rec.sim = sim;
        rec.flags = fl;
        rec.pass = cos_exceeds(cb, pa, pb, prm.cos_num, prm.cos_den) ? 1 : 0;
        *dst = rec;
    }
    __syncthreads();
}

// shared memory of exact_body
template <int NW, int SMAX>
constexpr size_t exact_smem() {
    // rasters (odd row stride), keys[32], R and C bounds (2 x (2 SMAX + 1)), L and the task count (+ 2 pad), the
    // order and its buckets, profiles [2][2N] u16, row starts, each warp's segments
    constexpr size_t tasks = (2 * SMAX + 1) * (2 * ((SMAX + 7) / 8) + 1), N = 64 * NW;
    return 2 * 16 * N * ((NW / 2) | 1) + 32 * 8 + 4 * (2 * (2 * SMAX + 1) + 4) + 4 * (tasks + 1 + kBuckets) + 2 * 4 * N +
           4 * 2 * (N / 32) + exact_threads<NW>() / 32 * 2 * (2 * N + 2);
}

}  // namespace exact_dev
}  // namespace pcl
