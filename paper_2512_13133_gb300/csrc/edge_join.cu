// a2, edge gates: the self-join screen of all pairs i < j through E2 and E1
// (Sec. 2.2.2, Sec. 3.1 stage 1), 32 pairs per bit operation.
//
// A pair survives when its clips pass E2 (equal polygon counts, no border
// edge: bbox sizes within 2 tol) and, at the pre-alignment, every polygon of
// the smaller clip overlaps exactly one polygon of the larger one, no two the
// same (E1).  E1 needs every polygon of the smaller clip to meet an occupied
// cell of the larger clip's 64 x 64 grid; that necessary condition is tested
// for whole words of 32 larger clips at a time:
//
//  * Order the clips by (polygon count, index); of a pair the earlier one is
//    the smaller clip u, the later one the larger clip v.
//  * Subtiles: the clips, sorted by strips of bbox centre x and then by centre
//    y, in groups of 256 (8 words of 32; inside a group by (count, index), so
//    the members after u are a suffix).  For a group the bit table holds, per
//    cell, which members occupy it, and the same ORed over 1, 2, 4, 8 cells in
//    x times 1, 2, 4, 8 cells in y: 16 x 4096 cells x 32 bytes = 2 MB.
//  * A polygon of u lies in v's frame at a shift that depends on both centres
//    (half their difference, clamped to the marker).  Over the members of a
//    group it lies in an interval; the cells under the polygon moved by the
//    whole interval contain the cells of every member's shift, so a member
//    whose bits are zero there cannot pass.  At 100,000 clips the interval
//    adds about 12 dbu per axis to polygons of 20-120 dbu.  Any rectangle of
//    up to 16 x 16 cells is the union of four (overlapping) table entries.
//  * A warp takes one u and four groups, lane = (group, word): one 32-byte
//    sector of table per group and entry.  Lane (group, j) prepares the table
//    positions of polygons j, j + 8, ... (ascending area, so that most members
//    fall away early) and they are handed round by shuffles.
//
// The pairs left (0.3 % of all; the exact grid test per pair would leave
// 0.25 %) go to a list, and edge_pair_check_kernel decides E2 and the exact
// correspondence, a warp per pair; pairs past the list's end are decided by
// the warp that found them.  The gate counts need no visit of the rejected
// pairs: E2's rejections are counted among the clips of equal polygon count
// without border edges, and E1 is all pairs minus the survivors minus E2.
//
// Bound: issue slots, table reads (mostly from L2) and their latency together.
// 100,000 clips of 256x256 px (5.0e9 pairs), one GB300: 10.0 ms a call - the
// screen 5.7 ms, the exact check of 15 M pairs 3.1 ms, the tables (0.8 GB
// written, 134 MB held) 0.26 ms, the sort and E2 0.2 ms - against 78.6 ms for
// the screen of pairs one by one in tiles (edge.cu), which stays for shards of
// the pair space, two clip sets and the topological pre-screen.  At 1,000
// clips the two take the same 0.1 ms.  Measured on the way: a table per group
// instead of per four interleaved groups 7.6 ms for the screen (more L1 tags
// per read), one polygon at a time 11.0 ms and two 6.1 (latency), 5 or 8 CTAs
// per SM 6.4 and 6.5 ms with two, entries for every width of 1 to 8 cells (half the
// reads, twice the tables) 6.4 ms with two and 6.0 with four, eight groups per warp
// with the lower words read only where they have members 6.4 ms; the check
// without the next pair's loads in flight 3.7 ms.
#include <type_traits>

#include "edge_dev.cuh"

namespace pcl {

namespace {
using namespace edge_dev;

constexpr int kSub = 256;                     // clips per group
constexpr uint32_t kCells = 16u * 4096u;      // table entries: (level in y, level in x, cell row, cell column)
constexpr uint32_t kQuadWords = (kCells + 1) * 32;  // u32 words of four groups' tables (8 MB), one entry of ones last
constexpr int kBatch = 64;                    // groups whose tables are held at a time
constexpr int kBins = 1024;                   // centre bins per axis, polygon-count bins
constexpr int kXPad = 72;                     // columns of a staged grid row (64 + 8 zeros)

struct GroupInfo {   // of one group of 256 clips
    int4 range;      // lowest and highest centre sum of the members that have x (y) edges: {cxlo, cxhi, cylo, cyhi}
    uint32_t flags;  // bit 0: some member has no x edges, bit 1: no y edges
    uint16_t first[64];  // position of the first member of at least k polygons
};

struct JoinWs {
    unsigned long long *local;  // [0] survivors, [1] E2 rejections
    unsigned int *n_empty;      // clips without polygons
    unsigned long long *n_list; // [batches] listed pairs
    uint32_t *hx, *he, *h2;     // histograms, then offsets: centre x, polygon count, (strip, centre y)
    int4 *uinfo;                // [n] {rectangle offset, count | has_x << 30 | has_y << 31, centre sums}
    int4 *poly8;                // [n * 8] the first eight polygons of each clip in area order
    uint32_t *order;            // [n] clips by (strip, centre y)
    uint32_t *empty;            // [n]
    int4 *erec;                 // [n] {count, bbox width, bbox height, 0} of clips without border edges, by count
    uint32_t *mem;              // [kBatch * 256] members of the batch's groups, in (count, index) order
    GroupInfo *info;            // [kBatch]
    uint2 *list;                // pairs (u, v) for the exact check
    uint32_t *tab;              // bit tables of the batch
    uint32_t list_cap;
    uint32_t n, groups, batch, strips;
};

__host__ __device__ inline uint32_t join_groups(uint32_t n) { return (n + kSub - 1) / kSub; }

// one list entry per 128 (clip, member) pairs of a batch, between 2^19 and
// 2^23: below about 1,000 clips the list holds every pair
uint32_t join_list_cap(uint32_t n) {
    const uint64_t c = (uint64_t)n * (n < kBatch * kSub ? n : kBatch * kSub) / 128;
    return c < (1u << 19) ? (1u << 19) : c > (1u << 23) ? (1u << 23) : (uint32_t)c;
}

size_t up(size_t v) { return (v + 255) & ~(size_t)255; }

// the parts of the workspace; returns the bytes (ws may be NULL)
size_t join_layout(uint32_t n, char *ws, JoinWs &w) {
    w.n = n;
    w.groups = join_groups(n);
    w.batch = w.groups < kBatch ? w.groups : kBatch;
    uint32_t s = 1;  // strips x groups per strip about square
    while ((s + 1) * (s + 1) <= w.groups) ++s;
    w.strips = s;
    w.list_cap = join_list_cap(n);
    const uint32_t batches = (w.groups + kBatch - 1) / kBatch;
    size_t o = 0;
    auto part = [&](auto *&p, size_t bytes) {
        p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(ws + o);
        o += up(bytes);
    };
    part(w.local, 64);
    part(w.n_empty, 64);
    part(w.n_list, 8 * (size_t)batches);
    part(w.hx, 4 * kBins);
    part(w.he, 4 * kBins);
    part(w.h2, 4 * (size_t)kBins * s);  // the parts so far start as zeros
    part(w.uinfo, 16 * (size_t)n);
    part(w.poly8, 16 * 8 * (size_t)n);
    part(w.order, 4 * (size_t)n);
    part(w.empty, 4 * (size_t)n);
    part(w.erec, 16 * (size_t)n);
    part(w.mem, 4 * (size_t)kSub * w.batch);
    part(w.info, sizeof(GroupInfo) * (size_t)w.batch);
    part(w.list, 8 * (size_t)w.list_cap);
    part(w.tab, 4 * (size_t)kQuadWords * ((w.batch + 3) / 4));
    return o;
}

__device__ __forceinline__ int centre_bin(int c, int W) {  // centre sums of [0, 2 W] in kBins bins
    const int v = (int)((long long)c * (kBins / 2) / W);
    return min(max(v, 0), kBins - 1);
}

__device__ __forceinline__ bool has_x(const int4 &i) { return (i.y >> 30) & 1; }
__device__ __forceinline__ bool has_y(const int4 &i) { return i.y < 0; }
__device__ __forceinline__ int polygons(const int4 &i) { return i.y & 0x3fffffff; }

// ---- the sort: per clip, its centre and counts
__device__ __forceinline__ void prep_clip(const pcl_clipset &cs, const JoinWs &w, uint32_t i, int W) {
    const int4 *e4 = reinterpret_cast<const int4 *>(cs.esig + (size_t)i * 8);
    const int4 lo = __ldg(e4), hi = __ldg(e4 + 1);  // {n, hasx, lox, hix}, {hasy, loy, hiy, border}
    const uint32_t off = __ldg(cs.rect_off + i);
    for (int k = 0; k < 8 && k < lo.x; ++k)
        w.poly8[(size_t)i * 8 + k] = __ldg(reinterpret_cast<const int4 *>(cs.rects) + off + __ldg(cs.rorder + off + k));
    w.uinfo[i] = make_int4((int)off, lo.x | (lo.y ? 1 << 30 : 0) | (hi.x ? (int)0x80000000 : 0),
                           lo.z + lo.w, hi.y + hi.z);
    atomicAdd(w.hx + centre_bin(lo.z + lo.w, W), 1u);
    if (lo.x == 0) w.empty[atomicAdd(w.n_empty, 1u)] = i;
    else if (!hi.w) atomicAdd(w.he + min(lo.x, kBins - 1), 1u);
}
__device__ __forceinline__ uint32_t strip_bin(const JoinWs &w, uint32_t i, int W) {
    const int4 u = w.uinfo[i];
    const uint32_t s = (uint32_t)((uint64_t)w.hx[centre_bin(u.z, W)] * w.strips / w.n);
    return min(s, w.strips - 1) * kBins + centre_bin(u.w, W);
}
__device__ __forceinline__ void place_clip(const pcl_clipset &cs, const JoinWs &w, uint32_t i, int W) {
    w.order[atomicAdd(w.h2 + strip_bin(w, i, W), 1u)] = i;
    const int4 *e4 = reinterpret_cast<const int4 *>(cs.esig + (size_t)i * 8);
    const int4 lo = __ldg(e4), hi = __ldg(e4 + 1);
    if (lo.x > 0 && !hi.w)
        w.erec[atomicAdd(w.he + min(lo.x, kBins - 1), 1u)] = make_int4(lo.x, lo.w - lo.z, hi.z - hi.y, 0);
}

__global__ void __launch_bounds__(256) join_prep_kernel(pcl_clipset cs, JoinWs w, int W) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.n; i += gridDim.x * blockDim.x)
        prep_clip(cs, w, i, W);
}
__global__ void __launch_bounds__(1024) join_scan_kernel(JoinWs w, int second) {
    if (second) {
        cta_scan(w.h2, w.h2, w.strips * kBins);
    } else {
        cta_scan(w.hx, w.hx, kBins);
        cta_scan(w.he, w.he, kBins);
    }
}
__global__ void __launch_bounds__(256) join_strip_kernel(JoinWs w, int W) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.n; i += gridDim.x * blockDim.x)
        atomicAdd(w.h2 + strip_bin(w, i, W), 1u);
}
__global__ void __launch_bounds__(256) join_place_kernel(pcl_clipset cs, JoinWs w, int W) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.n; i += gridDim.x * blockDim.x)
        place_clip(cs, w, i, W);
}
// the same steps in one CTA: for small sets the launches cost more than the work
__global__ void __launch_bounds__(1024) join_sort_small_kernel(pcl_clipset cs, JoinWs w, int W) {
    for (uint32_t i = threadIdx.x; i < w.n; i += 1024) prep_clip(cs, w, i, W);
    __syncthreads();
    cta_scan(w.hx, w.hx, kBins);
    cta_scan(w.he, w.he, kBins);
    for (uint32_t i = threadIdx.x; i < w.n; i += 1024) atomicAdd(w.h2 + strip_bin(w, i, W), 1u);
    __syncthreads();
    cta_scan(w.h2, w.h2, w.strips * kBins);
    for (uint32_t i = threadIdx.x; i < w.n; i += 1024) place_clip(cs, w, i, W);
}

// Rejections of E2 (a warp per clip, lanes over the clips after it in its count
// bin; only where gate counts are asked for), and the pairs of clips without polygons
// (similar by definition).  After the sort he[b] is the end of count bin b.  (A
// thread per clip left most of the GPU idle where all clips have one polygon
// count: 8,192 clips, 1.35 ms a call against 0.47.)
__global__ void __launch_bounds__(256) join_e2_kernel(JoinWs w, int tol, bool rejections, pcl_pair *out, uint64_t cap,
                                                      unsigned long long *count) {
    const uint32_t m = rejections ? w.he[kBins - 1] : 0u;
    const uint32_t lane = threadIdx.x & 31;
    unsigned long long rej = 0;
    for (uint32_t p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < m; p += (gridDim.x * blockDim.x) >> 5) {
        const int4 a = w.erec[p];
        const uint32_t end = w.he[min(a.x, kBins - 1)];
        uint32_t r = 0;
        for (uint32_t q = p + 1 + lane; q < end; q += 32) {
            const int4 b = w.erec[q];
            r += (a.x == b.x && (abs(a.y - b.y) > 2 * tol || abs(a.z - b.z) > 2 * tol)) ? 1u : 0u;
        }
        rej += r;
    }
    for (int o = 16; o; o >>= 1) rej += __shfl_xor_sync(0xffffffffu, rej, o);
    if ((threadIdx.x & 31) == 0 && rej) atomicAdd(w.local + 1, rej);
    const uint32_t e = *w.n_empty;
    if (e < 2) return;
    unsigned long long kept = 0;
    for (uint32_t p = blockIdx.x; p + 1 < e; p += gridDim.x) {
        const uint32_t a = w.empty[p];
        for (uint32_t q = p + 1 + threadIdx.x; q < e; q += blockDim.x) {
            const uint32_t b = w.empty[q];
            const unsigned long long at = atomicAdd(count, 1ull);
            if (at < cap) out[at] = pcl_pair{min(a, b), max(a, b)};
            ++kept;
        }
    }
    if (kept) atomicAdd(w.local, kept);
}

// The bit tables of one batch: CTA (g, quarter) sorts the group's members and
// writes the table entries of cell rows [16 quarter, 16 quarter + 16) from the
// grids' rows [16 quarter, +24) transposed into shared memory.
constexpr size_t kBuildSmem = 24 * kXPad * 8 * 4;

__global__ void __launch_bounds__(512) join_build_kernel(pcl_clipset cs, JoinWs w, uint32_t g0) {
    extern __shared__ __align__(16) uint32_t base[];  // [24][kXPad][8]
    __shared__ unsigned long long key[kSub];
    __shared__ uint32_t mem[kSub];
    __shared__ int red[8][8];
    const uint32_t gl = blockIdx.x >> 2, g = g0 + gl;
    const int quarter = blockIdx.x & 3, y0 = 16 * quarter;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t p = g * kSub + t;
    uint32_t id = 0xffffffffu;
    int4 ui = make_int4(0, 0, 0, 0);
    if (t < kSub) {
        if (p < w.n) {
            id = w.order[p];
            ui = w.uinfo[id];
        }
        // members past the set's end come last (the index keeps keys distinct)
        key[t] = p < w.n ? ((unsigned long long)polygons(ui) << 32) | id : (0x7fffffffull << 32) | (uint32_t)t;
    }
    for (int q = t; q < 24 * kXPad * 8; q += 512) base[q] = 0u;
    __syncthreads();
    if (t < kSub) {
        const unsigned long long k = key[t];
        int rank = 0;
        for (int q = 0; q < kSub; ++q) rank += key[q] < k ? 1 : 0;
        mem[rank] = id;
        if (quarter == 0) {
            w.mem[gl * kSub + rank] = id;
            const bool v = p < w.n && polygons(ui) > 0, vx = v && has_x(ui), vy = v && has_y(ui);
            const int r0 = __reduce_min_sync(0xffffffffu, vx ? ui.z : INT_MAX);
            const int r1 = __reduce_max_sync(0xffffffffu, vx ? ui.z : INT_MIN);
            const int r2 = __reduce_min_sync(0xffffffffu, vy ? ui.w : INT_MAX);
            const int r3 = __reduce_max_sync(0xffffffffu, vy ? ui.w : INT_MIN);
            const int r4 = (int)__reduce_or_sync(0xffffffffu, v ? (vx ? 0u : 1u) | (vy ? 0u : 2u) : 0u);
            if (lane == 0) {
                red[warp][0] = r0;
                red[warp][1] = r1;
                red[warp][2] = r2;
                red[warp][3] = r3;
                red[warp][4] = r4;
            }
        }
    }
    __syncthreads();
    if (quarter == 0) {
        GroupInfo *o = w.info + gl;
        if (t == 0) {
            int4 r = make_int4(INT_MAX, INT_MIN, INT_MAX, INT_MIN);
            int f = 0;
            for (int k = 0; k < 8; ++k) {
                r.x = min(r.x, red[k][0]);
                r.y = max(r.y, red[k][1]);
                r.z = min(r.z, red[k][2]);
                r.w = max(r.w, red[k][3]);
                f |= red[k][4];
            }
            o->range = r;
            o->flags = (uint32_t)f;
        }
        if (t < 64) {  // members past the set's end count as none: the suffix ends before them by their zero bits
            int c = 0;
            for (int q = 0; q < kSub; ++q) c += (int)(key[q] >> 32) < t ? 1 : 0;
            o->first[t] = (uint16_t)c;
        }
    }
    // transpose: task (word, 4 grid rows), lane = member
    for (int task = warp; task < 8 * 6; task += 16) {
        const int wd = task / 6, r0 = y0 + 4 * (task % 6);
        if (r0 >= 64) continue;
        const uint32_t m = mem[32 * wd + lane];
        ulonglong2 a = make_ulonglong2(0ull, 0ull), b = a;
        if (m != 0xffffffffu) {
            const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(cs.occ + (size_t)m * 64 + r0);
            a = __ldg(src);
            b = __ldg(src + 1);
        }
        const unsigned long long row[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t *d = base + (size_t)(r0 - y0 + k) * kXPad * 8 + wd;
            d[lane * 8] = transpose32((uint32_t)row[k], lane);
            d[(32 + lane) * 8] = transpose32((uint32_t)(row[k] >> 32), lane);
        }
    }
    __syncthreads();
    // thread (x, word): rows from the top down; v[l] the entry of 2^l cells in
    // x, and per l the last rows' entries of 1, 2 and 4 cells in y
    uint32_t *tab = w.tab + (size_t)(gl >> 2) * kQuadWords + 8 * (gl & 3) + (t & 7);
    if (quarter == 0 && t < 8) tab[(size_t)kCells * 32] = 0xffffffffu;
    uint32_t h1[4] = {0, 0, 0, 0}, h2[4][2] = {}, h4[4][4] = {};
#pragma unroll 4
    for (int r = 23; r >= 0; --r) {
        const uint32_t *s = base + (size_t)r * kXPad * 8 + t;
        uint32_t v[4];
        v[0] = s[0];
        v[1] = v[0] | s[8];
        v[2] = v[1] | s[16] | s[24];
        v[3] = v[2] | s[32] | s[40] | s[48] | s[56];
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            const uint32_t y2 = v[l] | h1[l];
            const uint32_t y4 = y2 | h2[l][1];
            const uint32_t y8 = y4 | h4[l][3];
            h1[l] = v[l];
            h2[l][1] = h2[l][0];
            h2[l][0] = y2;
            h4[l][3] = h4[l][2];
            h4[l][2] = h4[l][1];
            h4[l][1] = h4[l][0];
            h4[l][0] = y4;
            if (r < 16) {
                uint32_t *d = tab + (size_t)(l * 4096 + (y0 + r) * 64 + (t >> 3)) * 32;
                d[0] = v[l];
                d[(size_t)4 * 4096 * 32] = y2;
                d[(size_t)8 * 4096 * 32] = y4;
                d[(size_t)12 * 4096 * 32] = y8;
            }
        }
    }
}

__device__ __forceinline__ int half_trunc(int v) { return (v + (int)((unsigned)v >> 31)) >> 1; }  // v / 2

// E2 and the exact correspondence of one pair, u the smaller clip (warp-uniform)
__device__ __forceinline__ bool warp_pair_check(const pcl_params &prm, const pcl_clipset &cs, uint32_t u, uint32_t v,
                                                int lane) {
    const int4 *eu = reinterpret_cast<const int4 *>(cs.esig + (size_t)u * 8);
    const int4 *ev = reinterpret_cast<const int4 *>(cs.esig + (size_t)v * 8);
    const int4 ul = __ldg(eu), uh = __ldg(eu + 1), vl = __ldg(ev), vh = __ldg(ev + 1);
    const int offu = (int)__ldg(cs.rect_off + u), offv = (int)__ldg(cs.rect_off + v);
    const int tol = prm.edge_tol_dbu, M = prm.marker_dbu;
    if (ul.x == vl.x && !uh.w && !vh.w &&
        (abs((ul.w - ul.z) - (vl.w - vl.z)) > 2 * tol || abs((uh.z - uh.y) - (vh.z - vh.y)) > 2 * tol))
        return false;
    // the shift of u's polygons into v's frame (the pre-alignment is odd in
    // swapping the clips, so it does not matter which one is the pair's first)
    const int tx = ul.y && vl.y ? clampi(half_trunc((ul.z + ul.w) - (vl.z + vl.w)), -M, M) : 0;
    const int ty = uh.x && vh.x ? clampi(half_trunc((uh.y + uh.z) - (vh.y + vh.z)), -M, M) : 0;
    const int4 *r4 = reinterpret_cast<const int4 *>(cs.rects);
    return warp_correspond(r4 + offu, cs.rorder + offu, ul.x, r4 + offv, vl.x, true, tx, ty, lane);
}

// decide up to 32 pairs held by the lanes [0, m) and emit the survivors
__device__ __forceinline__ uint32_t warp_check_pairs(const pcl_params &prm, const pcl_clipset &cs, uint2 mine, int m,
                                                     pcl_pair *out, uint64_t cap, unsigned long long *count,
                                                     int lane) {
    unsigned ok = 0u;
    for (int q = 0; q < m; ++q) {
        const uint32_t u = __shfl_sync(0xffffffffu, mine.x, q), v = __shfl_sync(0xffffffffu, mine.y, q);
        if (warp_pair_check(prm, cs, u, v, lane)) ok |= 1u << q;
    }
    emit_pair(out, cap, count, (ok >> lane) & 1u, min(mine.x, mine.y), max(mine.x, mine.y));
    return (uint32_t)__popc(ok);
}

// out of line: rarely reached from the screen, whose registers it would raise
__device__ __noinline__ uint32_t check_pairs_here(const pcl_params &prm, const pcl_clipset &cs, uint2 mine, int m,
                                                  pcl_pair *out, uint64_t cap, unsigned long long *count, int lane) {
    return warp_check_pairs(prm, cs, mine, m, out, cap, count, lane);
}

constexpr int kQueuePairs = 64;

// cell of coordinate v; csh >= 0: the cell side is 1 << csh
__device__ __forceinline__ int grid_cell(int v, int csz, int csh) { return cell_of(v, csz, csh); }

// Table position of the cells [x0, x1] x [y0, y1]: the four entries lie at a
// byte offset x (of the entry; the lane's word is added by the reader), and
// further by (y & 15) entries in x, by the bytes of y's bits from 13 up in y
// (64 entries a row), and by both; kWide: more than 16 cells in x or y.
constexpr uint32_t kWide = 1u << 12;
__device__ __forceinline__ uint2 table_place(int x0, int y0, int x1, int y1) {
    const int wx = x1 - x0 + 1, wy = y1 - y0 + 1;  // >= 1
    const int lx = min(31 - __clz(wx), 3), ly = min(31 - __clz(wy), 3);
    const uint32_t dx = (uint32_t)(wx - (1 << lx)), dy = (uint32_t)(wy - (1 << ly));  // <= 8 up to 16 cells
    return make_uint2((uint32_t)((ly * 4 + lx) * 4096 + y0 * 64 + x0) * 128u,
                      dy << 13 | (wx > 16 || wy > 16 ? kWide : 0u) | (dx < 15u ? dx : 15u));
}

// One CTA: the clips u of a chunk, one per warp at a time, against four groups,
// lane = (group, word).  The groups' members sit in shared memory.
__global__ void __launch_bounds__(256, 6) join_screen_kernel(pcl_params prm, pcl_clipset cs, JoinWs w, uint32_t g0,
                                                             uint32_t n_groups, uint32_t chunk, uint32_t n_chunks,
                                                             uint32_t b, pcl_pair *out, uint64_t cap,
                                                             unsigned long long *count) {
    __shared__ uint2 queue[8][kQueuePairs];
    __shared__ uint2 member[4 * kSub];  // {clip, polygons}
    __shared__ uint16_t first[4][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sg = lane >> 3, wd = lane & 7;
    const uint32_t quad = blockIdx.x / n_chunks, ch = blockIdx.x % n_chunks;
    const uint32_t gl = quad * 4 + sg;
    const bool live = gl < n_groups;
    for (int t = threadIdx.x; t < 4 * kSub; t += blockDim.x) {
        const uint32_t v = quad * 4 + t / kSub < n_groups ? w.mem[quad * 4 * kSub + t] : 0xffffffffu;
        member[t] = make_uint2(v, v != 0xffffffffu ? (uint32_t)polygons(w.uinfo[v]) : 0u);
    }
    for (int t = threadIdx.x; t < 4 * 64; t += blockDim.x)
        first[t >> 6][t & 63] =
            quad * 4 + (t >> 6) < n_groups ? w.info[quad * 4 + (t >> 6)].first[t & 63] : (uint16_t)kSub;
    const char *tab = reinterpret_cast<const char *>(w.tab + (size_t)quad * kQuadWords);
    auto entry = [&](uint32_t o) { return __ldg(reinterpret_cast<const uint32_t *>(tab + o)); };
    const int4 range = w.info[live ? gl : 0].range;
    const uint32_t flags = w.info[live ? gl : 0].flags;
    __syncthreads();
    const int W = prm.window_dbu, M = prm.marker_dbu, csz = W / 64;
    const int csh = (csz & (csz - 1)) == 0 ? __ffs(csz) - 1 : -1;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t qn = 0, kept = 0;
    auto flush = [&](uint32_t m) {  // the first m (<= 32) queued pairs
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(w.n_list + b, (unsigned long long)m);
        at = __shfl_sync(0xffffffffu, at, 0);
        const uint2 e = queue[warp][lane];
        const uint32_t room = at < w.list_cap ? min(m, w.list_cap - (uint32_t)at) : 0u;
        if ((uint32_t)lane < room) w.list[at + lane] = e;
        if (room < m) {  // past the list's end: decide them here
            const int src = (int)min((uint32_t)lane + room, 31u);
            const uint2 r = make_uint2(__shfl_sync(0xffffffffu, e.x, src), __shfl_sync(0xffffffffu, e.y, src));
            kept += check_pairs_here(prm, cs, r, (int)(m - room), out, cap, count, lane);
        }
    };
    const uint32_t word = 4u * lane;  // this lane's word of a table entry
    // the members whose bit is set under the rectangle at place (x, y)
    auto covered = [&](uint32_t x, uint32_t y) -> uint32_t {
        const uint32_t o = x + word, ox = o + ((y & 15u) << 7), dy = y & ~8191u;
        return (entry(o) | entry(ox)) | (entry(o + dy) | entry(ox + dy));
    };
    // the same for a rectangle of any size: the level's entries side by side
    auto covered_wide = [&](uint32_t x, uint32_t y, uint32_t box) -> uint32_t {
        if (!(y & kWide)) return covered(x, y);
        const int x0 = box & 255, x1 = (box >> 8) & 255, y0 = (box >> 16) & 255, y1 = box >> 24;
        const uint32_t lev = x >> 19;
        const int sx = 1 << (lev & 3), sy = 1 << (lev >> 2);
        uint32_t acc = 0u;
        for (int r = y0;; r = min(r + sy, y1 + 1 - sy)) {
            for (int c = x0;; c = min(c + sx, x1 + 1 - sx)) {
                acc |= entry((lev * 4096u + (uint32_t)(r * 64 + c)) * 128u + word);
                if (c + sx > x1) break;
            }
            if (r + sy > y1) break;
        }
        return acc;
    };
    const int4 none = make_int4(0, 0, 0, 0);
    const uint32_t u1 = min(w.n, (ch + 1) * chunk);
    uint32_t u = ch * chunk + warp;
    int4 next = u < u1 ? w.uinfo[u] : none, qnext = u < u1 ? w.poly8[(size_t)u * 8 + wd] : none;
    for (; u < u1; u += 8) {
        const int4 ui = next;
        int4 q = qnext;
        if (u + 8 < u1) {  // the warp's next clip loads while this one is tested
            next = w.uinfo[u + 8];
            qnext = w.poly8[(size_t)(u + 8) * 8 + wd];
        }
        const int nu = polygons(ui);
        if (nu == 0) continue;
        // members of at least nu polygons: a suffix (those before u by index
        // are dropped when a pair is taken)
        const int pos = (int)first[sg][min(nu, 63)] - 32 * wd;
        uint32_t m = pos <= 0 ? 0xffffffffu : pos >= 32 ? 0u : 0xffffffffu << pos;
        if (!__any_sync(0xffffffffu, m != 0u)) continue;
        // shifts of u's polygons into the members' frames
        int dx0 = 0, dx1 = 0, dy0 = 0, dy1 = 0;
        if (has_x(ui) && range.x <= range.y) {
            dx0 = clampi(half_trunc(range.x - ui.z), -M, M);
            dx1 = clampi(half_trunc(range.y - ui.z), -M, M);
            if (flags & 1u) dx0 = min(dx0, 0), dx1 = max(dx1, 0);
        }
        if (has_y(ui) && range.z <= range.w) {
            dy0 = clampi(half_trunc(range.z - ui.w), -M, M);
            dy1 = clampi(half_trunc(range.w - ui.w), -M, M);
            if (flags & 2u) dy0 = min(dy0, 0), dy1 = max(dy1, 0);
        }
        for (int k0 = 0;;) {
            uint2 place = make_uint2(kCells * 128u, 0u);  // the entry of ones: no test
            uint32_t box = 0u;
            if (k0 + wd < nu && q.z > q.x && q.w > q.y) {
                const int x0 = grid_cell(q.x + dx0, csz, csh), x1 = grid_cell(q.z - 1 + dx1, csz, csh);
                const int y0 = grid_cell(q.y + dy0, csz, csh), y1 = grid_cell(q.w - 1 + dy1, csz, csh);
                place = table_place(x0, y0, x1, y1);
                box = (uint32_t)(x0 | x1 << 8 | y0 << 16 | y1 << 24);
            }
            const bool wide = __any_sync(0xffffffffu, place.y & kWide);
            bool any = true;
            // four polygons at a time: sixteen independent loads (past the last polygon: the entry of ones)
            for (int k = 0; k < 8 && k0 + k < nu; k += 4) {
                uint32_t x[4], y[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    x[j] = __shfl_sync(0xffffffffu, place.x, (lane & 24) | (k + j));
                    y[j] = __shfl_sync(0xffffffffu, place.y, (lane & 24) | (k + j));
                }
                if (!wide) {
                    if (m) m &= (covered(x[0], y[0]) & covered(x[1], y[1])) & (covered(x[2], y[2]) & covered(x[3], y[3]));
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t bj = __shfl_sync(0xffffffffu, box, (lane & 24) | (k + j));
                        if (m) m &= covered_wide(x[j], y[j], bj);
                    }
                }
                any = __any_sync(0xffffffffu, m != 0u);
                if (!any) break;
            }
            k0 += 8;
            if (!any || k0 >= nu) break;
            if (k0 + wd < nu)
                q = __ldg(reinterpret_cast<const int4 *>(cs.rects) + ui.x + __ldg(cs.rorder + ui.x + k0 + wd));
        }
        // the pairs left: members after u in (count, index) order
        while (__any_sync(0xffffffffu, m != 0u)) {
            uint2 v = make_uint2(0u, 0u);
            bool keep = false;
            if (m) {
                v = member[32 * lane + __ffs(m) - 1];
                m &= m - 1u;
                keep = v.x != 0xffffffffu && ((int)v.y > nu || ((int)v.y == nu && v.x > u));
            }
            const unsigned kb = __ballot_sync(0xffffffffu, keep);
            if (!kb) continue;
            if (keep) queue[warp][qn + __popc(kb & lt)] = make_uint2(u, v.x);
            qn += (uint32_t)__popc(kb);
            __syncwarp();
            if (qn >= 32) {
                flush(32);
                __syncwarp();
                uint2 e = make_uint2(0u, 0u);
                if ((uint32_t)lane + 32 < qn) e = queue[warp][lane + 32];
                __syncwarp();
                if ((uint32_t)lane + 32 < qn) queue[warp][lane] = e;
                qn -= 32;
                __syncwarp();
            }
        }
    }
    if (qn) flush(qn);
    if (lane == 0 && kept) atomicAdd(w.local, (unsigned long long)kept);
}

// The listed pairs, up to 32 per warp at a time: lane q reads the signatures of pair
// q and decides E2; the correspondence takes the pairs one by one with the
// whole warp, as warp_correspond does, the next pair's polygons (the larger
// clip's, and the first eight of the smaller one) loading while one is tested.
__global__ void __launch_bounds__(256, 4) edge_pair_check_kernel(pcl_params prm, pcl_clipset cs, JoinWs w, uint32_t b,
                                                                 pcl_pair *out, uint64_t cap,
                                                                 unsigned long long *count) {
    const unsigned full = 0xffffffffu;
    const unsigned long long listed = w.n_list[b];
    const uint32_t n = listed < w.list_cap ? (uint32_t)listed : w.list_cap;
    const int lane = threadIdx.x & 31;
    const uint32_t w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const int4 *r4 = reinterpret_cast<const int4 *>(cs.rects);
    const int4 none = make_int4(0, 0, 0, 0);
    const int tol = prm.edge_tol_dbu, M = prm.marker_dbu;
    unsigned long long kept = 0;
    const uint32_t per = min(32u, (n + nw - 1) / nw);  // a short list is spread over all warps
    for (uint32_t t0 = w0 * per; t0 < n; t0 += nw * per) {  // warp-uniform
        uint2 mine = make_uint2(0u, 0u);
        int offu = 0, nu = 0, offv = 0, nv = 0, tx = 0, ty = 0;
        bool take = (uint32_t)lane < per && t0 + lane < n;
        if (take) {
            mine = w.list[t0 + lane];
            const int4 *eu = reinterpret_cast<const int4 *>(cs.esig + (size_t)mine.x * 8);
            const int4 *ev = reinterpret_cast<const int4 *>(cs.esig + (size_t)mine.y * 8);
            const int4 ul = __ldg(eu), uh = __ldg(eu + 1), vl = __ldg(ev), vh = __ldg(ev + 1);
            offu = (int)__ldg(cs.rect_off + mine.x);
            offv = (int)__ldg(cs.rect_off + mine.y);
            nu = ul.x;
            nv = vl.x;
            take = !(nu == nv && !uh.w && !vh.w &&
                     (abs((ul.w - ul.z) - (vl.w - vl.z)) > 2 * tol || abs((uh.z - uh.y) - (vh.z - vh.y)) > 2 * tol));
            tx = ul.y && vl.y ? clampi(half_trunc((ul.z + ul.w) - (vl.z + vl.w)), -M, M) : 0;
            ty = uh.x && vh.x ? clampi(half_trunc((uh.y + uh.z) - (vh.y + vh.z)), -M, M) : 0;
        }
        unsigned todo = __ballot_sync(full, take), ok = 0u;
        int4 l0n = none, l1n = none, sn = none;  // the next pair's polygons
        auto fetch = [&](int q) {
            const int ov = __shfl_sync(full, offv, q), cv = __shfl_sync(full, nv, q), cu = __shfl_sync(full, nu, q);
            const uint32_t u = __shfl_sync(full, mine.x, q);
            l0n = lane < cv ? __ldg(r4 + ov + lane) : none;
            l1n = lane + 32 < cv ? __ldg(r4 + ov + lane + 32) : none;
            sn = lane < min(cu, 8) ? w.poly8[(size_t)u * 8 + lane] : none;
        };
        if (todo) fetch(__ffs(todo) - 1);
        while (todo) {
            const int q = __ffs(todo) - 1;
            todo &= todo - 1u;
            int4 l0 = l0n, l1 = l1n, s = sn;
            if (todo) fetch(__ffs(todo) - 1);
            const int cu = __shfl_sync(full, nu, q), cv = __shfl_sync(full, nv, q), ou = __shfl_sync(full, offu, q);
            const int px = __shfl_sync(full, tx, q), py = __shfl_sync(full, ty, q);
            bool good = true;
            if (cv > 64) {
                const int ov = __shfl_sync(full, offv, q);
                good = warp_correspond(r4 + ou, cs.rorder + ou, cu, r4 + ov, cv, true, px, py, lane);
            } else {
                l0 = make_int4(l0.x + px, l0.y + py, l0.z + px, l0.w + py);
                l1 = make_int4(l1.x + px, l1.y + py, l1.z + px, l1.w + py);
                const bool v0 = lane < cv, v1 = lane + 32 < cv;
                int c0 = 0, c1 = 0;
                for (int k0 = 0, kn = min(cu, 8); good && kn > 0;) {
                    if (cv <= 32) {
                        for (int k = 0; k < kn; ++k) {
                            const int sx0 = __shfl_sync(full, s.x, k), sy0 = __shfl_sync(full, s.y, k);
                            const int sx1 = __shfl_sync(full, s.z, k), sy1 = __shfl_sync(full, s.w, k);
                            const bool h0 = v0 && sx0 < l0.z && l0.x < sx1 && sy0 < l0.w && l0.y < sy1;
                            const unsigned b0 = __ballot_sync(full, h0);
                            good = b0 != 0u && !(b0 & (b0 - 1u));  // exactly one partner
                            if (!good) break;
                            c0 += h0 ? 1 : 0;
                        }
                    } else {
                        for (int k = 0; k < kn; ++k) {
                            const int sx0 = __shfl_sync(full, s.x, k), sy0 = __shfl_sync(full, s.y, k);
                            const int sx1 = __shfl_sync(full, s.z, k), sy1 = __shfl_sync(full, s.w, k);
                            const bool h0 = v0 && sx0 < l0.z && l0.x < sx1 && sy0 < l0.w && l0.y < sy1;
                            const bool h1 = v1 && sx0 < l1.z && l1.x < sx1 && sy0 < l1.w && l1.y < sy1;
                            good = __popc(__ballot_sync(full, h0)) + __popc(__ballot_sync(full, h1)) == 1;
                            if (!good) break;
                            c0 += h0 ? 1 : 0;
                            c1 += h1 ? 1 : 0;
                        }
                    }
                    // the polygons after the first eight, 32 at a time
                    k0 += k0 ? 32 : 8;
                    kn = min(cu - k0, 32);
                    if (good && kn > 0) s = lane < kn ? __ldg(r4 + ou + __ldg(cs.rorder + ou + k0 + lane)) : none;
                }
                good = good && !__any_sync(full, c0 > 1 || c1 > 1);
            }
            if (good) ok |= 1u << q;
        }
        emit_pair(out, cap, count, (ok >> lane) & 1u, min(mine.x, mine.y), max(mine.x, mine.y));
        kept += (unsigned long long)__popc(ok);
    }
    if (lane == 0 && kept) atomicAdd(w.local, kept);
}

__global__ void join_gates_kernel(JoinWs w, unsigned long long *gates) {
    const unsigned long long n = w.n, total = n * (n - 1) / 2, kept = w.local[0], e2 = w.local[1];
    gates[0] += kept;
    gates[PCL_GATE_E2_BBOX] += e2;
    gates[PCL_GATE_E1_MATCH] += total - kept - e2;
}

}  // namespace

size_t edge_join_workspace(uint32_t n) {
    JoinWs w;
    return join_layout(n, nullptr, w);
}

cudaError_t launch_edge_join(const pcl_params &prm, const pcl_clipset &cs, void *ws, size_t ws_bytes, pcl_pair *out,
                             uint64_t cap, unsigned long long *count, unsigned long long *gates, int num_sms,
                             cudaStream_t st) {
    const uint32_t n = cs.n_clips;
    if (n < 2) return cudaSuccess;
    JoinWs w;
    if (!ws || ws_bytes < join_layout(n, static_cast<char *>(ws), w)) return cudaErrorInvalidValue;
    const int W = prm.window_dbu;
    cudaError_t e = cudaMemsetAsync(ws, 0, (size_t)(reinterpret_cast<char *>(w.uinfo) - static_cast<char *>(ws)), st);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(join_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBuildSmem);
    if (e != cudaSuccess) return e;
    if (n <= 8192) {
        join_sort_small_kernel<<<1, 1024, 0, st>>>(cs, w, W);
    } else {
        const unsigned grid = (unsigned)min((n + 255) / 256, (uint32_t)num_sms * 8);
        join_prep_kernel<<<grid, 256, 0, st>>>(cs, w, W);
        join_scan_kernel<<<1, 1024, 0, st>>>(w, 0);
        join_strip_kernel<<<grid, 256, 0, st>>>(w, W);
        join_scan_kernel<<<1, 1024, 0, st>>>(w, 1);
        join_place_kernel<<<grid, 256, 0, st>>>(cs, w, W);
    }
    join_e2_kernel<<<(unsigned)min((n + 7) / 8, (uint32_t)num_sms * 8), 256, 0, st>>>(w, prm.edge_tol_dbu,
                                                                                     gates != nullptr, out, cap, count);
    for (uint32_t g0 = 0, b = 0; g0 < w.groups; g0 += w.batch, ++b) {
        const uint32_t ng = min(w.batch, w.groups - g0), quads = (ng + 3) / 4;
        join_build_kernel<<<4 * ng, 512, kBuildSmem, st>>>(cs, w, g0);
        // clips per CTA (eight warps): enough CTAs to fill the GPU a few times over
        uint32_t chunk = (uint32_t)((uint64_t)n * quads / ((uint64_t)num_sms * 16)) & ~7u;
        chunk = chunk < 8 ? 8 : chunk > 512 ? 512 : chunk;
        const uint32_t n_chunks = (n + chunk - 1) / chunk;
        join_screen_kernel<<<quads * n_chunks, 256, 0, st>>>(prm, cs, w, g0, ng, chunk, n_chunks, b, out, cap, count);
        edge_pair_check_kernel<<<num_sms * 8, 256, 0, st>>>(prm, cs, w, b, out, cap, count);
    }
    if (gates) join_gates_kernel<<<1, 1, 0, st>>>(w, gates);
    return cudaGetLastError();
}

}  // namespace pcl
