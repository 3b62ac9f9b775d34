// The exact windowed correlation of two clips from their rectangles (Sec. 2.2.1,
// Eq. 2: c(s) = sum_x A(x) B(x - s) for the shifts of the marker window).
//
// When no two rectangles of a clip share a pixel, the raster is the sum of the
// rectangles' pixel ranges and c is the sum over pairs (rectangle of A,
// rectangle of B) of fx(dx) fy(dy), where on each axis
//   f(d) = max(0, min(a1, b1 + d) - max(a0, b0 + d))
// is a trapezoid: piecewise linear with four breakpoints.  Its second
// difference over the window d = -S .. S (zeros before it) has at most six
// non-zero entries (the first two values and a +-1 at each breakpoint inside),
// so a pair of rectangles adds at most 36 products to a K x K table (K = 2S + 1),
// and two prefix sums along each axis turn the table into c(s) for every shift,
// in integers (mod 2^32; c itself is below 2^18).  A pair of
// clips costs a few thousand warp instructions instead of a popcount per shift,
// row and word.  Bound by issue slots and, at about 16 warps an SM, latency.
//
// One warp per pair of clips.  Clips of more than kRectMax rectangles, whose
// rectangles share pixels, or whose rectangles are not the raster's (a caller may
// have written the buffer again: the rasters are what a record is about), are
// left to the callers' other paths: the ranges must be disjoint, every pixel of
// theirs set, and their areas add up to the raster's ones.  That look takes a
// third of the instructions where it is taken per pair, so long lists take it per
// clip (verdicts, below).
//
// One GB300, same-seed pairs of clips of 21 rectangles, a call: 12,001 pairs of
// 512x512 px 0.21 ms (0.19 without any look at the rasters) against 4.2 ms for their window
// scan, 100,000 of 256x256 px 0.66 ms (0.63) against 6.5 (scan) and 21 ms (FP16
// tensor cores, full items).
#pragma once

#include "common.cuh"

namespace pcl {
namespace rect_corr {

constexpr int kRectMax = 64;
constexpr uint16_t kRectPending = 0xffff;  // flags of a record that another kernel still has to write

// pixel range of an edge pair: first index whose centre p i + p/2 is >= v,
// ceil((2 v - p) / (2 p)), clamped to [lo, hi]; psh >= 0: the pitch is 1 << psh
__device__ __forceinline__ int pix_index(int v, int p, int psh, int lo, int hi) {
    long long q;
    if (psh >= 0) {
        q = (2LL * v + p - 1) >> (psh + 1);
    } else {
        const long long a = 2LL * v - p, b = 2LL * p;
        q = a / b;
        if (a % b != 0 && a > 0) ++q;
    }
    return (int)(q < lo ? lo : q > hi ? hi : q);
}

// a set's rectangles can be read (cosine libraries of a server may come without)
__host__ __device__ inline bool has_rects(const pcl_clipset &cs) {
    return cs.rect_off && cs.rects && (reinterpret_cast<uintptr_t>(cs.rects) & 15u) == 0;
}

// Per-warp shared memory: the table (K x K int, K odd: rows and columns spread
// over the banks), both clips' pixel ranges {x0, x1, y0, y1}, and a queue of
// rectangle pairs.
struct Scratch {
    int *table;
    short4 *ra, *rb;
    uint16_t *queue;  // [64]
};
__host__ __device__ inline size_t scratch_bytes(int S) {
    const int K = 2 * S + 1;
    return ((size_t)4 * K * K + 2 * 8 * kRectMax + 2 * 64 + 15) & ~(size_t)15;
}
__device__ __forceinline__ Scratch scratch_at(unsigned char *base, int S) {
    const int K = 2 * S + 1;
    Scratch s;
    s.ra = reinterpret_cast<short4 *>(base);
    s.rb = s.ra + kRectMax;
    s.queue = reinterpret_cast<uint16_t *>(s.rb + kRectMax);
    s.table = reinterpret_cast<int *>(s.queue + 64);
    (void)K;
    return s;
}

// stage a clip's n <= kRectMax rectangles as pixel ranges clamped to [lo, hi)
// on both axes; returns the pixels of all ranges (warp-uniform)
__device__ __forceinline__ uint32_t stage_rects(const int4 *rects, int n, int p, int psh, int lo, int hi, short4 *dst,
                                                int lane) {
    uint32_t area = 0;
    for (int t = lane; t < n; t += 32) {
        const int4 q = __ldg(rects + t);
        const int x0 = pix_index(q.x, p, psh, lo, hi), x1 = pix_index(q.z, p, psh, lo, hi);
        const int y0 = pix_index(q.y, p, psh, lo, hi), y1 = pix_index(q.w, p, psh, lo, hi);
        const bool some = x0 < x1 && y0 < y1;
        dst[t] = some ? make_short4((short)x0, (short)x1, (short)y0, (short)y1) : make_short4(0, 0, 0, 0);
        area += some ? (uint32_t)(x1 - x0) * (uint32_t)(y1 - y0) : 0u;
    }
    return __reduce_add_sync(0xffffffffu, area);
}

// no two of the n staged ranges share a pixel (an empty range, (0, 0, 0, 0), has
// none): lane i compares range i with the n / 2 ranges after it, past the last
// one from the first on
__device__ __forceinline__ bool ranges_disjoint(const short4 *r, int n, int lane) {
    bool shared_px = false;
    for (int i = lane; i - lane < n; i += 32) {
        const short4 a = i < n ? r[i] : make_short4(0, 0, 0, 0);
        int j = i;
#pragma unroll 4
        for (int d = 0; d < n / 2; ++d) {
            j = j + 1 < n ? j + 1 : 0;
            const short4 b = r[j];
            shared_px |= (max(a.x, b.x) < min(a.y, b.y)) & (max(a.z, b.z) < min(a.w, b.w));
        }
    }
    return !__any_sync(0xffffffffu, shared_px);
}

// every pixel of the n staged ranges is set in the raster: rows of nw words, the
// pixel (x, y) at bit x + o of row y + o.  Eight lanes per rectangle, four of its
// rows per lane at a time, the first and the last word of each: eight loads in
// flight.  With 32 lanes per rectangle, a word and a rectangle after the other, it
// took longer than the tables: 12,000 pairs of 40 rectangles 401 us at 256x256 px and 988
// at 512x512, now 240 and 619, without any look at the raster 167 and 282.
__device__ __forceinline__ bool ranges_set(const short4 *r, int n, const uint64_t *__restrict__ bits, int nw, int o,
                                           int lane) {
    uint64_t unset = 0ull;
    bool wide = false;  // some rectangle covers a word between its first and its last
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 4) {
        const int i = i0 + (lane >> 3), sub = lane & 7;
        const short4 q = i < n ? r[i] : make_short4(0, 0, 0, 0);
        const int x0 = q.x + o, x1 = q.y + o - 1, w0 = x0 >> 6, w1 = x1 >> 6;
        uint64_t first = ~0ull << (x0 & 63), last = ~0ull >> (63 - (x1 & 63));
        const bool two = w1 > w0;
        if (!two) first &= last, last = 0ull;
        wide |= w1 > w0 + 1;
        const int rows = __reduce_max_sync(0xffffffffu, q.w - q.z), mine = q.w - q.z - sub;
        const uint64_t *p = bits + (q.z + sub + o) * nw + w0;
#pragma unroll 1
        for (int y = 0; y < rows; y += 32, p += 32 * nw) {
            uint64_t a[4], b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool in = y + 8 * j < mine;
                a[j] = in ? __ldg(p + 8 * j * nw) : ~0ull;
                b[j] = in && two ? __ldg(p + 8 * j * nw + (w1 - w0)) : ~0ull;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) unset |= (~a[j] & first) | (~b[j] & last);
        }
    }
    if (__any_sync(0xffffffffu, wide)) {
        for (int i = 0; i < n; ++i) {
            const short4 q = r[i];
            for (int y = q.z + lane; y < q.w; y += 32)
                for (int w = ((q.x + o) >> 6) + 1; w < (q.y + o - 1) >> 6; ++w) unset |= ~__ldg(bits + (y + o) * nw + w);
        }
    }
    return !__any_sync(0xffffffffu, unset != 0ull);
}

// the n staged ranges share no pixel, and all of theirs are set in the raster.  Out
// of line: it is needed for both clips, and its code beside the tables' in a
// kernel twice costs instruction fetches (a quarter of the stalls)
static __device__ __noinline__ bool ranges_in_raster(const short4 *r, int n, const uint64_t *__restrict__ bits, int nw,
                                                     int o, int lane) {
    return ranges_disjoint(r, n, lane) && ranges_set(r, n, bits, nw, o, lane);
}

// the entries of f's second difference on one axis: position in [0, 2S] and weight (0: none)
__device__ __forceinline__ void trapezoid(int a0, int a1, int b0, int b1, int S, int (&q)[6], int (&w)[6]) {
    const int f0 = max(0, min(a1, b1 - S) - max(a0, b0 - S));
    const int f1 = max(0, min(a1, b1 - S + 1) - max(a0, b0 - S + 1));
    q[0] = 0;
    w[0] = f0;
    q[1] = 1;
    w[1] = S > 0 ? f1 - 2 * f0 : 0;
    const int t[4] = {a0 - b1, a0 - b0, a1 - b1, a1 - b0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int at = t[k] + 1 + S;
        const bool in = at >= 2 && at <= 2 * S;
        q[2 + k] = in ? at : 0;
        w[2 + k] = in ? (k == 0 || k == 3 ? 1 : -1) : 0;
    }
}

// c(dx, dy) for every shift of the window, from the staged ranges: visit(c, dx,
// dy) is called once per shift, by the lane that holds it.
template <typename Visit>
__device__ __forceinline__ void rect_surface(const Scratch &s, int na, int nb, int S, int lane, Visit visit) {
    const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
    const int K = 2 * S + 1;
    for (int t = lane; t < K * K; t += 32) s.table[t] = 0;
    __syncwarp();  // also orders the staged ranges
    auto add = [&](int code) {
        const short4 a = s.ra[code >> 6], b = s.rb[code & 63];
        int qx[6], wx[6], qy[6], wy[6];
        trapezoid(a.x, a.y, b.x, b.y, S, qx, wx);
        trapezoid(a.z, a.w, b.z, b.w, S, qy, wy);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            if (wy[i] == 0) continue;
            int *row = s.table + qy[i] * K;
#pragma unroll
            for (int j = 0; j < 6; ++j)
                if (wx[j] != 0) atomicAdd(row + qx[j], wx[j] * wy[i]);
        }
    };
    // rectangle pairs that meet at some shift of the window, 32 at a time
    int n = 0;
    for (int i = 0; i < na; ++i) {
        const short4 a = s.ra[i];
        for (int j0 = 0; j0 < nb; j0 += 32) {
            const int j = j0 + lane;
            const short4 b = j < nb ? s.rb[j] : make_short4(0, 0, 0, 0);
            const bool hit = a.x < b.y + S && b.x - S < a.y && a.z < b.w + S && b.z - S < a.w && b.x < b.y && a.x < a.y;
            const unsigned m = __ballot_sync(full, hit);
            if (!m) continue;
            if (hit) s.queue[n + __popc(m & lt)] = (uint16_t)(i << 6 | j);
            n += __popc(m);
            __syncwarp();
            if (n >= 32) {
                add(s.queue[lane]);
                __syncwarp();
                const int rest = lane + 32 < n ? s.queue[lane + 32] : 0;
                __syncwarp();
                if (lane + 32 < n) s.queue[lane] = (uint16_t)rest;
                n -= 32;
                __syncwarp();
            }
        }
    }
    if (lane < n) add(s.queue[lane]);
    __syncwarp();
    // two prefix sums along x, a lane per row (a single row past a multiple of
    // 32 by warp scans)
    auto scan2 = [&](int v) {  // the lanes' values summed twice
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(full, v, o);
                if (lane >= o) v += t;
            }
        return v;
    };
    const bool odd_one = K > 32 && K % 32 == 1;
    const int whole = odd_one ? K - 1 : K;
    for (int y = lane; y < whole; y += 32) {
        int *row = s.table + y * K;
        int s1 = 0, s2 = 0;
#pragma unroll 4
        for (int x = 0; x < K; ++x) {
            s1 += row[x];
            s2 += s1;
            row[x] = s2;
        }
    }
    if (odd_one) {
        int *row = s.table + (K - 1) * K;
        int c1 = 0, c2 = 0;  // once and twice summed values before this stretch
        for (int x0 = 0; x0 < K; x0 += 32) {
            const int v = x0 + lane < K ? row[x0 + lane] : 0;
            int one = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(full, one, o);
                if (lane >= o) one += t;
            }
            const int two = scan2(v) + c2 + c1 * (lane + 1);
            if (x0 + lane < K) row[x0 + lane] = two;
            c2 = __shfl_sync(full, two, 31);
            c1 += __shfl_sync(full, one, 31);
        }
    }
    __syncwarp();
    // along y, a lane per column
    for (int x = lane; x < whole; x += 32) {
        const int *col = s.table + x;
        int s1 = 0, s2 = 0;
#pragma unroll 4
        for (int y = 0; y < K; ++y) {
            s1 += col[y * K];
            s2 += s1;
            visit((uint32_t)s2, x - S, y - S);
        }
    }
    if (odd_one) {
        const int *col = s.table + K - 1;
        int c1 = 0, c2 = 0;
        for (int y0 = 0; y0 < K; y0 += 32) {
            const int v = y0 + lane < K ? col[(y0 + lane) * K] : 0;
            int one = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(full, one, o);
                if (lane >= o) one += t;
            }
            const int two = scan2(v) + c2 + c1 * (lane + 1);
            if (y0 + lane < K) visit((uint32_t)two, S, y0 + lane - S);
            c2 = __shfl_sync(full, two, 31);
            c1 += __shfl_sync(full, one, 31);
        }
    }
    __syncwarp();  // the scratch is free again
}

// the n staged ranges are the window raster of clip c of set cs, whose pixels
// they number `area`, and share none
__device__ __forceinline__ bool ranges_are_raster(const short4 *r, int n, uint32_t area, const pcl_clipset &cs,
                                                  uint32_t c, const Geo &g, int lane) {
    return area == cs.pop[c] && ranges_in_raster(r, n, cs.bits + (size_t)c * g.N * g.nw, g.nw, 0, lane);
}

// Verdicts: where a list has at least twice as many pairs as its sets have clips, each
// clip is compared with its raster once, before the pairs.  The verdicts wait in
// the records that the call is to write, 32 clips in the first bytes of each, until a kernel has
// left each pair's in the last word of its own record (`reserved`): a call needs no
// workspace for them and may run beside others on other streams.  A call, with a look
// per pair and with verdicts: 100,000 pairs of 20,000 clips of 256x256 px 1.03 and 0.66 ms,
// 12,001 of 2,600 of 512x512 px 0.26 and 0.21 ms, re-extraction of 60,000 pairs of
// 12,200 clips 1.15 and 0.91 ms.  Short lists would pay more for the two launches.
__host__ __device__ inline bool verdicts_pay(uint64_t pairs, uint64_t clips) { return pairs >= 4096 && pairs >= 2 * clips; }
__device__ __forceinline__ unsigned char *verdict_at(pcl_record *out, uint64_t clip) {
    return reinterpret_cast<unsigned char *>(out + clip / 32) + clip % 32;
}
__host__ __device__ inline bool one_set(const pcl_clipset &a, const pcl_clipset &b) {
    return a.n_clips == b.n_clips && a.bits == b.bits && a.pop == b.pop && a.rects == b.rects && a.rect_off == b.rect_off;
}

// whether the rectangles of clip c are its window raster; staged into r (one warp)
__device__ __forceinline__ bool window_verdict(const pcl_clipset &cs, uint32_t c, const Geo &g, int psh, short4 *r,
                                               int lane) {
    const uint32_t o = __ldg(cs.rect_off + c);
    const int n = (int)(__ldg(cs.rect_off + c + 1) - o);
    if (n < 0 || n > kRectMax) return false;
    __syncwarp();  // the previous clip's ranges are no longer read
    const uint32_t area = stage_rects(reinterpret_cast<const int4 *>(cs.rects) + o, n, g.p, psh, 0, g.N, r, lane);
    __syncwarp();
    return ranges_are_raster(r, n, area, cs, c, g, lane);
}

// each pair's verdict from its clips' (set B's follow from base_b on); clips: of both sets
template <typename Record>
__global__ void __launch_bounds__(256) pair_verdict_kernel(uint32_t n_a, uint32_t n_b, uint64_t base_b, uint64_t clips,
                                                           const pcl_pair *pairs, uint64_t n,
                                                           const unsigned long long *d_n, Record *out) {
    if (d_n && *d_n < n) n = *d_n;
    if (!verdicts_pay(n, clips)) return;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (uint64_t)gridDim.x * blockDim.x) {
        const pcl_pair pr = pairs[t];
        out[t].reserved = pr.a < n_a && pr.b < n_b && *verdict_at(out, pr.a) && *verdict_at(out, base_b + pr.b) ? 1u : 0u;
    }
}

// Whether the pair takes this path: few enough rectangles, and (after staging)
// ranges that are the rasters.  Stages both clips.  verdict: that of the pair, -1 if
// there is none yet.
__device__ __forceinline__ bool stage_pair(const pcl_clipset &A, const pcl_clipset &B, const pcl_pair pr, const Geo &g,
                                           int psh, const Scratch &s, int verdict, int &na, int &nb, int lane) {
    if (verdict == 0) return false;
    const uint32_t oa = __ldg(A.rect_off + pr.a), ob = __ldg(B.rect_off + pr.b);
    na = (int)(__ldg(A.rect_off + pr.a + 1) - oa);
    nb = (int)(__ldg(B.rect_off + pr.b + 1) - ob);
    if (na < 0 || nb < 0 || na > kRectMax || nb > kRectMax) return false;
    __syncwarp();  // the scratch's previous contents are no longer read
    const uint32_t aa = stage_rects(reinterpret_cast<const int4 *>(A.rects) + oa, na, g.p, psh, 0, g.N, s.ra, lane);
    const uint32_t ab = stage_rects(reinterpret_cast<const int4 *>(B.rects) + ob, nb, g.p, psh, 0, g.N, s.rb, lane);
    __syncwarp();
    return verdict > 0 ||
           (ranges_are_raster(s.ra, na, aa, A, pr.a, g, lane) && ranges_are_raster(s.rb, nb, ab, B, pr.b, g, lane));
}

// The cosine record of one pair by the exact argmax (one warp; lane 0 writes
// it): what the exact window scan and the tensor-core correlation give.  false:
// the pair does not take this path, nothing is written.
__device__ __forceinline__ bool rect_record(const pcl_params &prm, const Geo &g, int psh, const pcl_clipset &A,
                                            const pcl_clipset &B, const pcl_pair pr, const Scratch &s,
                                            int verdict, pcl_record *dst, int lane) {
    int na, nb;
    if (!stage_pair(A, B, pr, g, psh, s, verdict, na, nb, lane)) return false;
    const int S = g.S;
    // best by (c, then smaller |dx| + |dy|, smaller dy, smaller dx): shift_key's order
    uint32_t bc = 0, bt = 0;
    rect_surface(s, na, nb, S, lane, [&](uint32_t c, int dx, int dy) {
        if (c >= bc) {
            const uint32_t t = (uint32_t)shift_key(0, dx, dy, S);
            if (c > bc || t > bt) {
                bc = c;
                bt = t;
            }
        }
    });
    const uint32_t cb = __reduce_max_sync(0xffffffffu, bc);
    const uint32_t tb = __reduce_max_sync(0xffffffffu, bc == cb ? bt : 0u);
    if (lane == 0) {
        const int dx = S - (int)(tb & 0xffu), dy = S - (int)((tb >> 8) & 0xffu);
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
    return true;
}

}  // namespace rect_corr
}  // namespace pcl
