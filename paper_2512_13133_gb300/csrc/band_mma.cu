// a2, cosine gates at 256x256 and 512x512 px: the band join's density gate (G3)
// as a matrix product on the 5th-generation tensor cores.
//
// G3 bounds the overlap by sum_k min(cnt_A(k), nbr_B(k)) over the 16x16 blocks
// (gates.cu).  With thresholds t_0 = 0 < t_1 < .. < t_L (t_L = 256, a block's
// pixels) and B's sums rounded up to the next threshold,
//   min(cnt_A, nbr_B) <= sum_l f_l(cnt_A) [nbr_B > t_l],
//   f_l(a) = min(a, t_{l+1}) - min(a, t_l)  (a's share of the l-th segment),
// a product of one vector per representative with one 0/1 vector per member:
// a GEMM over all pairs of the band in E4M3 (f rounded up to its 4 significant
// bits) with FP32 accumulators, K = 16x16 blocks x L.  A pair whose product is at
// or below the largest overlap that fails Eq. 2 fails G3 as well; at 256x256 px
// and L = 4 that decides 99.4 % of the band (the exact sums of this direction
// would decide 99.7 %), and only the rest take the exact G3 and G2.
//
// band_feature_kernel writes both vectors per clip in area order, laid out as
// the MMA reads them (no-swizzle K-major core matrices, 8 rows x 16 bytes;
// panels of 128 representatives, blocks of 256 members), so that operands
// come by plain bulk copies.  band_mma_kernel, one CTA per SM: an item is a
// panel and up to kSeg member blocks of its band; the panel's vectors stay in
// shared memory, the blocks stream through a ring; one thread copies, one
// issues tcgen05.mma (128 x 256 x 32), four warps compare the accumulators
// (double buffered in tensor memory) with T sqrt(|A| |B|), a 32-column word of
// decisions per lane, and list the pairs left.  band_list_kernel decides those
// exactly, a warp per pair.  Should the list be too short (nearly identical
// clips) or a bounded wait run out, it is dropped and the band join (gates.cu,
// cross.cu) runs instead, as it does for smaller rasters, shards, the
// topological pre-screen and callers without workspace.
//
// 100,000 clips of 256x256 px (5.9e8 band pairs), one GB300: 1.5 ms a call - the
// products 0.68 ms (4.8 GB of operands from L2, 7.2 TB/s, which bounds them:
// the MMAs alone would take 0.27 ms), the exact check of 3.2 M pairs 0.68 ms,
// the vectors (205 MB) 0.07 ms, the sort 0.03 ms - against 21.5 ms for the band
// join's G3 on the CUDA cores.
#include <type_traits>

#include "gates.cuh"
#include "tc_dev.cuh"

namespace pcl {

namespace {
using namespace tc_dev;

constexpr int kPanel = 128, kBlock = 256;  // representatives (M) and members (N) of one MMA tile
constexpr int kStage = 32768;              // bytes of one ring stage: 256 members x 128 bytes of K
constexpr int kSeg = 16;                   // member blocks per item at most
constexpr int kMmaThreads = 256;
constexpr uint32_t kTmem = 512;
constexpr uint64_t kMaxList = 1u << 23;   // listed pairs at most
constexpr float kSlack = 1.0f - 1.0f / 1024.0f;  // on T sqrt(|A| |B|): float rounding, with room to spare

// K bytes per clip: L thresholds of nb2 blocks, at most 1,024
__host__ __device__ inline int levels_of(int nb2) { return nb2 >= 1024 ? 1 : 4; }
__host__ __device__ inline int kbytes_of(int nb2) { return nb2 * levels_of(nb2); }
__host__ __device__ inline int threshold(int levels, int l) {  // t_l
    return l == 0 ? 0 : l >= levels ? 256 : 32 << (l - 1);     // 0, 32, 64, 128, 256
}

struct BandWs {
    unsigned long long *seen;   // band pairs
    unsigned long long *n_list; // listed pairs
    unsigned int *overflow;     // 1: the list was too short
    uint32_t *seg;              // member blocks per item
    uint32_t *item_off;         // [panels + 1]
    uint32_t *beg, *end;        // [rows] band of each representative, positions in the members' area order
    float *ra;                  // [rows] T sqrt(area) with the slack
    float *cb;                  // [blocks * 256] sqrt(area) of the members
    unsigned char *P, *Q;       // vectors: panels x K x 128 bytes, blocks x K x 256 bytes
    uint2 *list;                // positions (representative, member)
    const uint32_t *row_order, *row_pop, *col_order, *col_pop;  // the area orders
    uint32_t list_cap, rows, cols, panels, blocks;
    int kb;
};

size_t up(size_t v) { return (v + 255) & ~(size_t)255; }

// the parts of the workspace; with_cols: the members' vectors are part of it
// (and the bands of a self-join), otherwise Q, cb, beg and end are the caller's
size_t band_layout(const Geo &g, uint32_t rows, uint32_t cols, uint64_t list_cap, bool self, bool with_cols, char *ws,
                   BandWs &w) {
    w.rows = rows;
    w.cols = cols;
    w.panels = (rows + kPanel - 1) / kPanel;
    w.blocks = (cols + kBlock - 1) / kBlock;
    w.kb = kbytes_of(g.nb * g.nb);
    w.list_cap = list_cap < (1u << 12) ? (1u << 12) : list_cap > kMaxList ? (uint32_t)kMaxList : (uint32_t)list_cap;
    size_t o = 0;
    auto part = [&](auto *&p, size_t bytes) {
        p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(ws + o);
        o += up(bytes);
    };
    part(w.seen, 8);
    part(w.n_list, 8);
    part(w.overflow, 4);  // the parts so far start as zeros
    part(w.seg, 4);
    part(w.item_off, 4 * ((size_t)w.panels + 1));
    if (self) {
        part(w.beg, 4 * (size_t)rows);
        part(w.end, 4 * (size_t)rows);
    }
    part(w.ra, 4 * (size_t)rows);
    part(w.list, 8 * (size_t)w.list_cap);
    part(w.P, (size_t)w.panels * kPanel * w.kb);
    if (with_cols) {
        part(w.cb, 4 * (size_t)kBlock * w.blocks);
        part(w.Q, (size_t)w.blocks * kBlock * w.kb);
    }
    return o;
}

// listed pairs there is room for: the bound leaves 0.55 % of a band of about
// an eighth of the members; nearly identical clips leave more, and overflow.  A
// query's band also holds smaller members, of which the bound (its own counts against their
// sums) leaves more: room for 3 % of it, as with 1 % every request against
// 2,000,000 clips overflowed and took the band join after all.
uint64_t list_room(uint64_t rows, uint64_t cols, bool self) {
    const uint64_t c = self ? rows * cols / 512 : rows * (cols / 256 + 64);
    return self && c < (1u << 16) ? 1u << 16 : c;
}

// integer 0..256 as E4M3, rounded up to 4 significant bits
__device__ __forceinline__ uint32_t e4m3_up(int x) {
    if (x == 0) return 0u;
    int e = 31 - __clz(x);
    int m = e <= 3 ? x << (3 - e) : (x + (1 << (e - 3)) - 1) >> (e - 3);  // 8 .. 16
    if (m == 16) {
        ++e;
        m = 8;
    }
    return (uint32_t)(((e + 7) << 3) | (m & 7));
}

// Both vectors of 64 clips per CTA: a thread takes 16 blocks of one clip, looks
// their E4M3 codes up for all levels and writes 16 bytes per level and vector;
// 16 consecutive threads take consecutive clips, whose 16-byte rows of a core
// matrix are adjacent.  Positions past n are zeros (their products exceed no
// threshold).  (Converting every value for every level took 185 us at 100,000
// clips, the table 72 us.)
constexpr int kFeatureClips = 64;

// ROWS: the representatives' vectors, thresholds and (BANDS, the self-join)
// bands; COLS: the members' vectors.  order, spop: the set's area order; n clips.
template <int LV, bool ROWS, bool COLS, bool BANDS>
__global__ void __launch_bounds__(256) band_feature_kernel(pcl_params prm, pcl_clipset cs, BandWs w,
                                                           const uint32_t *order, const uint32_t *spop, uint32_t n,
                                                           const uint32_t *cum) {
    const Geo g = make_geo(prm);
    const int nb2 = g.nb * g.nb;
    // per block count 0..256: byte l is the code of its share of level l
    __shared__ uint32_t code[257];
    for (int a = threadIdx.x; a < 257; a += 256) {
        uint32_t c = 0u;
#pragma unroll
        for (int l = 0; l < LV; ++l)
            c |= e4m3_up(min(a, threshold(LV, l + 1)) - min(a, threshold(LV, l))) << (8 * l);
        code[a] = c;
    }
    __syncthreads();
    const int r = threadIdx.x & 15;
    for (int c0 = 0; c0 < kFeatureClips; c0 += 16) {
        const uint32_t p = blockIdx.x * kFeatureClips + c0 + r;
        const bool live = p < n;
        const uint32_t *cw = reinterpret_cast<const uint32_t *>(cs.blk + (size_t)(live ? order[p] : 0) * 2 * nb2);
        unsigned char *P = w.P + (size_t)(p / kPanel) * kPanel * w.kb + (p % kPanel) * 16;
        unsigned char *Q = w.Q + (size_t)(p / kBlock) * kBlock * w.kb + (p % kBlock) * 16;
        for (int j = threadIdx.x >> 4; j < nb2 / 16; j += 16) {
            uint32_t f[LV][4], q[LV][4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                uint32_t c[4], d[4];  // codes of four counts, and their neighbourhood sums
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const uint32_t x = live ? __ldg(cw + 8 * j + 2 * h + s) : 0u;
                    const uint32_t y = live ? __ldg(cw + nb2 / 2 + 8 * j + 2 * h + s) : 0u;
                    c[2 * s] = code[min(x & 0xffffu, 256u)];
                    c[2 * s + 1] = code[min(x >> 16, 256u)];
                    d[2 * s] = y & 0xffffu;
                    d[2 * s + 1] = y >> 16;
                }
#pragma unroll
                for (int l = 0; l < LV; ++l) {
                    const uint32_t t0 = (uint32_t)threshold(LV, l);
                    f[l][h] = q[l][h] = 0u;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        f[l][h] |= (c[e] >> (8 * l) & 0xffu) << (8 * e);
                        q[l][h] |= (d[e] > t0 ? 0x38u : 0u) << (8 * e);  // 1.0
                    }
                }
            }
#pragma unroll
            for (int l = 0; l < LV; ++l) {
                const size_t k = (size_t)(l * nb2 / 16 + j);  // 16-byte column of K
                if (ROWS && p < w.panels * kPanel)
                    *reinterpret_cast<uint4 *>(P + k * (16 * kPanel)) = make_uint4(f[l][0], f[l][1], f[l][2], f[l][3]);
                if (COLS && p < w.blocks * kBlock)
                    *reinterpret_cast<uint4 *>(Q + k * (16 * kBlock)) = make_uint4(q[l][0], q[l][1], q[l][2], q[l][3]);
            }
        }
    }
    if (threadIdx.x >= kFeatureClips) return;
    const uint32_t p = blockIdx.x * kFeatureClips + threadIdx.x;
    const float s = p < n ? sqrtf((float)spop[p]) : 0.0f;
    if (COLS && p < w.blocks * kBlock) w.cb[p] = s;
    if (ROWS) {
        unsigned long long band = 0;
        if (p < n) {
            w.ra[p] = s * ((float)prm.cos_num / (float)prm.cos_den) * kSlack;
            if (BANDS) {
                const uint64_t num2 = (uint64_t)prm.cos_num * prm.cos_num, den2 = (uint64_t)prm.cos_den * prm.cos_den;
                const uint64_t pa = spop[p], all = (uint64_t)g.N * g.N;
                uint64_t vmax = pa == 0 ? 0 : (den2 * pa - 1) / num2;
                if (vmax > all) vmax = all;
                w.beg[p] = p + 1;
                w.end[p] = cum[vmax + 1];
            }
            band = w.end[p] - w.beg[p];
        }
        for (int o = 16; o; o >>= 1) band += __shfl_xor_sync(0xffffffffu, band, o);
        if ((threadIdx.x & 31) == 0 && band) atomicAdd(w.seen, band);
    }
}

// first member block of a panel's band, and how many blocks it meets (begins
// and ends do not decrease along the area order)
__device__ __forceinline__ void panel_blocks(const BandWs &w, uint32_t panel, uint32_t &first, uint32_t &count) {
    const uint32_t p0 = panel * kPanel, last = min(w.rows, p0 + kPanel) - 1;
    const uint32_t b = w.beg[p0], e = w.end[last];
    first = b / kBlock;
    count = e > b ? (e + kBlock - 1) / kBlock - first : 0u;
}

// Items of the panels before each panel (one CTA): an item takes up to kSeg
// member blocks, fewer when that would leave SMs without an item.
__global__ void __launch_bounds__(1024) band_items_kernel(BandWs w, uint32_t num_sms) {
    __shared__ unsigned int tiles;
    if (threadIdx.x == 0) tiles = 0u;
    __syncthreads();
    unsigned int t = 0;
    for (uint32_t i = threadIdx.x; i < w.panels; i += 1024) {
        uint32_t f, c;
        panel_blocks(w, i, f, c);
        w.item_off[i] = c;
        t += c;
    }
    t = __reduce_add_sync(0xffffffffu, t);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(&tiles, t);
    __syncthreads();
    const uint32_t seg = min(max(tiles / (2 * num_sms), 1u), (uint32_t)kSeg);
    for (uint32_t i = threadIdx.x; i < w.panels; i += 1024) w.item_off[i] = (w.item_off[i] + seg - 1) / seg;
    __syncthreads();
    const uint32_t total = cta_scan(w.item_off, w.item_off, w.panels);
    if (threadIdx.x == 0) {
        w.item_off[w.panels] = total;
        *w.seg = seg;
    }
}

struct BandItem {
    uint32_t panel, first, count;  // member blocks [first, first + count)
};
__device__ __forceinline__ BandItem band_item(const BandWs &w, uint32_t it) {
    uint32_t lo = 0, hi = w.panels;  // the last panel with item_off <= it
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) / 2;
        if (w.item_off[mid] <= it) lo = mid;
        else hi = mid;
    }
    BandItem b;
    uint32_t f, c;
    panel_blocks(w, lo, f, c);
    const uint32_t seg = *w.seg, s = (it - w.item_off[lo]) * seg;
    b.panel = lo;
    b.first = f + s;
    b.count = min(c - s, seg);
    return b;
}

// barriers: panel full / empty, accumulators full[2] / empty[2], end, ring full[ST] / empty[ST]
enum { kPFull = 0, kPEmpty = 1, kAcc = 2, kAccFree = 4, kEnd = 6, kRing = 7 };

template <int KB>
struct BandSmem {
    static constexpr uint32_t panel = KB * kPanel;
    static constexpr int stages = (int)((232448u - panel - 4096u) / kStage) > 4 ? 4 : (int)((232448u - panel - 4096u) / kStage);
    static constexpr uint32_t ring = panel;
    static constexpr uint32_t queue = ring + stages * kStage;  // [4 warps][64] uint2
    static constexpr uint32_t bars = queue + 4 * 64 * 8;
    static constexpr uint32_t bytes = bars + (kRing + 2 * stages) * 8 + 16;
};

template <int KB>
__global__ void __launch_bounds__(kMmaThreads, 1) band_mma_kernel(BandWs w, unsigned long long wait_ns) {
    using SM = BandSmem<KB>;
    constexpr int ST = SM::stages, CH = KB / 128;  // ring stages, K chunks per member block
    extern __shared__ __align__(1024) unsigned char sm[];
    volatile uint32_t *misc = reinterpret_cast<volatile uint32_t *>(sm + SM::bars + (kRing + 2 * ST) * 8);
    const volatile uint32_t *abortf = misc + 1;
    const uint32_t sbase = smem_u32(sm), bar0 = sbase + SM::bars;
    auto bar = [&](int k) { return bar0 + 8u * (uint32_t)k; };
    // a wait that ran out gives the product up: the band join decides instead
    auto raise_abort = [&]() {
        misc[1] = 1u;
        *w.overflow = 1u;
    };
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(bar(kPFull), 1);
        mbar_init(bar(kPEmpty), 1);
        for (int k = 0; k < 2; ++k) {
            mbar_init(bar(kAcc + k), 1);
            mbar_init(bar(kAccFree + k), 128);
        }
        mbar_init(bar(kEnd), 1);
        for (int k = 0; k < ST; ++k) {
            mbar_init(bar(kRing + k), 1);
            mbar_init(bar(kRing + ST + k), 1);
        }
        misc[1] = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32((const void *)misc)),
                     "r"(kTmem));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = misc[0];
    const uint32_t n_items = w.item_off[w.panels];

    if (warp == 0) {
        // ---------------------------------------------------------------- copies
        if (lane == 0) {
            bool ok = true;
            uint32_t li = 0, e = 0, panels = 0;  // items, stages and panels so far
            for (uint32_t it = blockIdx.x; it < n_items && ok; it += gridDim.x, ++li) {
                const BandItem item = band_item(w, it);
                if (li && !(ok = wait_phase(bar(kPEmpty), (li - 1) & 1, abortf, wait_ns))) break;
                mbar_expect(bar(kPFull), SM::panel);
                const unsigned char *P = w.P + (size_t)item.panel * SM::panel;
                for (uint32_t o = 0; o < SM::panel; o += 16384) bulk_copy(sbase + o, P + o, 16384, bar(kPFull));
                ++panels;
                const unsigned char *Q = w.Q + (size_t)item.first * KB * kBlock;
                for (uint32_t s = 0; s < item.count * CH; ++s, ++e) {
                    const uint32_t k = e % ST;
                    if (e >= ST && !(ok = wait_phase(bar(kRing + ST + k), (e / ST - 1) & 1, abortf, wait_ns))) break;
                    mbar_expect(bar(kRing + k), kStage);
                    bulk_copy(sbase + SM::ring + k * kStage, Q + (size_t)s * kStage, kStage, bar(kRing + k));
                }
            }
            if (!ok) raise_abort();
            // every copy issued has landed before the shared memory is given up
            for (uint32_t k = 0; k < (uint32_t)ST && k < e; ++k) {
                const uint32_t last = (e - 1 - k) / ST * ST + k;  // the last use of stage k
                if (!wait_phase(bar(kRing + k), (last / ST) & 1, nullptr, kWaitNs)) raise_abort();
            }
            if (panels && !wait_phase(bar(kPFull), (panels - 1) & 1, nullptr, kWaitNs)) raise_abort();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issue
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_of(kPanel, kBlock, kOpE4M3);
            bool ok = true;
            uint32_t li = 0, e = 0, t = 0;  // items, stages, tiles so far
            for (uint32_t it = blockIdx.x; it < n_items && ok; it += gridDim.x, ++li) {
                const BandItem item = band_item(w, it);
                if (!(ok = wait_phase(bar(kPFull), li & 1, abortf, wait_ns))) break;
                for (uint32_t b = 0; b < item.count && ok; ++b, ++t) {
                    const uint32_t buf = t & 1;
                    if (t >= 2 && !(ok = wait_phase(bar(kAccFree + buf), ((t >> 1) - 1) & 1, abortf, wait_ns))) break;
                    fence_after();
                    for (int c = 0; c < CH; ++c, ++e) {
                        const uint32_t k = e % ST;
                        if (!(ok = wait_phase(bar(kRing + k), (e / ST) & 1, abortf, wait_ns))) break;
                        fence_after();
#pragma unroll
                        for (int s = 0; s < 4; ++s) {  // K = 32: two core matrices
                            const uint64_t ad = smem_desc(sbase + (uint32_t)(8 * c + 2 * s) * (16 * kPanel), 16 * kPanel, 128);
                            const uint64_t bd = smem_desc(sbase + SM::ring + k * kStage + (uint32_t)(2 * s) * (16 * kBlock),
                                                          16 * kBlock, 128);
                            mma<true>(tmem + buf * kBlock, ad, bd, idesc, (c | s) != 0 ? 1u : 0u);
                        }
                        mma_commit(bar(kRing + ST + k));
                    }
                    if (ok) mma_commit(bar(kAcc + buf));
                }
                if (ok) mma_commit(bar(kPEmpty));
            }
            if (!ok) raise_abort();
            // every MMA issued so far has completed before the tensor memory is released
            mma_commit(bar(kEnd));
            if (!wait_phase(bar(kEnd), 0, nullptr, kWaitNs)) raise_abort();
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ---------------------------------------------------------------- decisions
        const int quarter = warp & 3;
        uint2 *queue = reinterpret_cast<uint2 *>(sm + SM::queue) + quarter * 64;
        const unsigned lt = (1u << lane) - 1u;
        uint32_t qn = 0, t = 0;
        bool ok = true;
        auto flush = [&](uint32_t m) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(w.n_list, (unsigned long long)m);
            at = __shfl_sync(0xffffffffu, at, 0);
            if ((uint32_t)lane < m && at + lane < w.list_cap) w.list[at + lane] = queue[lane];
            if (lane == 0 && at + m > w.list_cap) *w.overflow = 1u;
        };
        for (uint32_t it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
            const BandItem item = band_item(w, it);
            const uint32_t p = item.panel * kPanel + 32 * quarter + lane;
            const uint32_t beg = p < w.rows ? w.beg[p] : 0u, end = p < w.rows ? w.end[p] : 0u;
            const float ra = w.ra[min(p, w.rows - 1)];
            for (uint32_t b = 0; b < item.count; ++b, ++t) {
                const uint32_t buf = t & 1;
                ok = wait_phase(bar(kAcc + buf), (t >> 1) & 1, abortf, wait_ns);
                if (__any_sync(0xffffffffu, !ok)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t q0 = (item.first + b) * kBlock;
                const uint32_t src = tmem + ((uint32_t)(32 * quarter) << 16) + buf * kBlock;
                for (int c = 0; c < kBlock; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(src + c, v);
                    const float4 *th = reinterpret_cast<const float4 *>(w.cb + q0 + c);
                    tmem_wait_ld();
                    uint32_t hit = 0u;  // bit 31 - j: v[j] above its threshold
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 s = __ldg(th + j / 4);
                        hit = __funnelshift_l(__float_as_uint(fmaf(ra, s.x, -__uint_as_float(v[j]))), hit, 1);
                        hit = __funnelshift_l(__float_as_uint(fmaf(ra, s.y, -__uint_as_float(v[j + 1]))), hit, 1);
                        hit = __funnelshift_l(__float_as_uint(fmaf(ra, s.z, -__uint_as_float(v[j + 2]))), hit, 1);
                        hit = __funnelshift_l(__float_as_uint(fmaf(ra, s.w, -__uint_as_float(v[j + 3]))), hit, 1);
                    }
                    hit = __brev(hit);
                    // members of the band
                    const int lo = (int)beg - (int)(q0 + c), hi = (int)end - (int)(q0 + c);
                    uint32_t in = hi >= 32 ? 0xffffffffu : hi <= 0 ? 0u : (1u << hi) - 1u;
                    in &= lo <= 0 ? 0xffffffffu : lo >= 32 ? 0u : 0xffffffffu << lo;
                    hit &= in;
                    while (__any_sync(0xffffffffu, hit != 0u)) {
                        const bool have = hit != 0u;
                        const unsigned hb = __ballot_sync(0xffffffffu, have);
                        if (have) {
                            queue[qn + __popc(hb & lt)] = make_uint2(p, q0 + c + __ffs(hit) - 1);
                            hit &= hit - 1u;
                        }
                        qn += (uint32_t)__popc(hb);
                        __syncwarp();
                        if (qn >= 32) {
                            flush(32);
                            __syncwarp();
                            uint2 r = make_uint2(0u, 0u);
                            if ((uint32_t)lane + 32 < qn) r = queue[lane + 32];
                            __syncwarp();
                            if ((uint32_t)lane + 32 < qn) queue[lane] = r;
                            qn -= 32;
                            __syncwarp();
                        }
                    }
                }
                fence_before();
                mbar_arrive(bar(kAccFree + buf));
            }
        }
        if (qn) flush(qn);
        if (!ok && lane == 0) raise_abort();
        __syncwarp();
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem));
}

// The listed pairs: exact G3, then G2, a warp per pair; and the pairs of empty
// clips.  A warp takes up to 32 pairs at a time: lane q reads pair q's clips and
// finds its threshold, then the pairs go one by one, the next pair's first 64
// blocks loading while one is tested (1.10 -> 0.68 ms at 100,000 clips).
// CROSS: representatives of set A (rows), members of set B; otherwise one set.
template <int NPL, bool CROSS>
__global__ void __launch_bounds__(256) band_list_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B, BandWs w,
                                                        pcl_pair *out, uint64_t cap, unsigned long long *count,
                                                        unsigned long long *local) {
    if (*w.overflow) return;
    extern __shared__ uint16_t g2_scratch[];
    const unsigned full = 0xffffffffu;
    const Geo g = make_geo(prm);
    const int lane = threadIdx.x & 31, nb2 = g.nb * g.nb, words = nb2 / 2;
    uint16_t *scratch = g2_scratch + (threadIdx.x >> 5) * 2 * (g.N + 2 * g.S + 32);
    const uint32_t n = (uint32_t)*w.n_list;
    const uint32_t w0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const uint32_t *blk_a = reinterpret_cast<const uint32_t *>(A.blk), *blk_b = reinterpret_cast<const uint32_t *>(B.blk);
    auto pair_of = [](uint32_t a, uint32_t b) { return CROSS ? pcl_pair{a, b} : pcl_pair{min(a, b), max(a, b)}; };
    unsigned long long kept = 0, g2 = 0;
    const uint32_t per = min(32u, (n + nw - 1) / nw);  // a short list (a request's) is spread over all warps
    for (uint32_t t0 = w0 * per; t0 < n; t0 += nw * per) {  // warp-uniform
        const int m = (int)min(n - t0, per);
        uint32_t a = 0, b = 0;
        int um = 0, pa = 0, pb = 0;  // areas are at most 512^2
        if (lane < m) {
            const uint2 e = w.list[t0 + lane];
            a = w.row_order[e.x];
            b = w.col_order[e.y];
            pa = (int)w.row_pop[e.x];
            pb = (int)w.col_pop[e.y];
            um = (int)cos_umax((uint64_t)pa, (uint64_t)pb, prm.cos_num, prm.cos_den);
        }
        uint32_t ca = 0, da = 0, cb = 0, db = 0;  // the next pair's first chunk: counts and neighbourhood sums
        auto fetch = [&](int q) {
            const uint32_t *x = blk_a + (size_t)__shfl_sync(full, a, q) * nb2;
            const uint32_t *y = blk_b + (size_t)__shfl_sync(full, b, q) * nb2;
            ca = __ldg(x + lane);
            da = __ldg(x + words + lane);
            cb = __ldg(y + lane);
            db = __ldg(y + words + lane);
        };
        fetch(0);
        for (int q = 0; q < m; ++q) {
            const uint32_t qa = __shfl_sync(full, a, q), qb = __shfl_sync(full, b, q);
            const int u = __shfl_sync(full, um, q);
            const int tA = __shfl_sync(full, pa, q) - u, tB = __shfl_sync(full, pb, q) - u;
            // G3: the deficits as warp_g3_rejects sums them, 64 blocks at a time
            uint32_t sa = __reduce_add_sync(full, ca - __vminu2(ca, db)), sb = __reduce_add_sync(full, cb - __vminu2(cb, da));
            if (q + 1 < m) fetch(q + 1);
            int DA = (int)((sa & 0xffffu) + (sa >> 16)), DB = (int)((sb & 0xffffu) + (sb >> 16));
            bool rej = DA >= tA || DB >= tB;
            const uint32_t *x = blk_a + (size_t)qa * nb2, *y = blk_b + (size_t)qb * nb2;
            for (int k = 32 + lane; !rej && k < words; k += 32) {  // words is a multiple of 32
                const uint32_t c0 = __ldg(x + k), d0 = __ldg(x + words + k), c1 = __ldg(y + k), d1 = __ldg(y + words + k);
                sa = __reduce_add_sync(full, c0 - __vminu2(c0, d1));
                sb = __reduce_add_sync(full, c1 - __vminu2(c1, d0));
                DA += (int)((sa & 0xffffu) + (sa >> 16));
                DB += (int)((sb & 0xffffu) + (sb >> 16));
                rej = DA >= tA || DB >= tB;
            }
            if (rej) continue;
            if (warp_g2_rejects_groups<NPL>(A.prof + (size_t)qa * 2 * g.N, B.prof + (size_t)qb * 2 * g.N, g.S,
                                            (int64_t)u, lane, scratch)) {
                ++g2;
                continue;
            }
            ++kept;
            if (lane == 0) {
                const unsigned long long at = atomicAdd(count, 1ull);
                if (at < cap) out[at] = pair_of(qa, qb);
            }
        }
    }
    // empty representatives (the first ones): their band holds the empty
    // members only, similar by definition
    for (uint32_t p = blockIdx.x; p < w.rows && w.row_pop[p] == 0; p += gridDim.x) {
        const uint32_t a = w.row_order[p], e = w.end[p];
        for (uint32_t q0 = w.beg[p]; q0 < e; q0 += blockDim.x) {
            const uint32_t q = q0 + threadIdx.x;
            const uint32_t b = q < e ? w.col_order[q] : 0u;
            const unsigned m = __ballot_sync(full, q < e);
            unsigned long long base = 0;
            if (lane == 0 && m) base = atomicAdd(count, (unsigned long long)__popc(m));
            base = __shfl_sync(full, base, 0);
            if (q < e && base + lane < cap) out[base + lane] = pair_of(a, b);
            kept += (unsigned long long)__popc(m);
        }
    }
    if (lane == 0) {
        if (kept) atomicAdd(local + 0, kept);
        if (g2) atomicAdd(local + PCL_GATE_G2_PROFILE, g2);
    }
}

// G3's rejections: the band's pairs that neither survived nor failed G2
__global__ void band_count_kernel(BandWs w, unsigned long long *local) {
    if (!*w.overflow) local[PCL_GATE_G3_DENSITY] = *w.seen - local[0] - local[PCL_GATE_G2_PROFILE];
}

template <int KB, int NPL, bool CROSS>
cudaError_t launch_t(const pcl_params &prm, const Geo &g, const pcl_clipset &A, const pcl_clipset &B, const BandWs &w,
                     pcl_pair *out, uint64_t cap, unsigned long long *count, unsigned long long *local, int num_sms,
                     unsigned long long wait_ns, cudaStream_t st) {
    band_items_kernel<<<1, 1024, 0, st>>>(w, (uint32_t)num_sms);
    const uint32_t bytes = BandSmem<KB>::bytes;
    cudaError_t e = cudaFuncSetAttribute(band_mma_kernel<KB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    band_mma_kernel<KB><<<num_sms, kMmaThreads, bytes, st>>>(w, wait_ns ? wait_ns : kWaitNs);
    const size_t scratch = 8 * 2 * 2 * (size_t)(g.N + 2 * g.S + 32);
    band_list_kernel<NPL, CROSS><<<num_sms * 8, 256, scratch, st>>>(prm, A, B, w, out, cap, count, local);
    band_count_kernel<<<1, 1, 0, st>>>(w, local);
    return cudaGetLastError();
}

template <bool ROWS, bool COLS, bool BANDS>
void features(const pcl_params &prm, const Geo &g, const pcl_clipset &cs, const BandWs &w, const uint32_t *order,
              const uint32_t *spop, uint32_t n, const uint32_t *cum, cudaStream_t st) {
    const uint32_t reach = COLS ? w.blocks * kBlock : w.panels * kPanel;  // COLS reaches at least as far as ROWS of one set
    const unsigned grid = (reach + kFeatureClips - 1) / kFeatureClips;
    if (grid == 0) return;
    if (g.N == 256) band_feature_kernel<4, ROWS, COLS, BANDS><<<grid, 256, 0, st>>>(prm, cs, w, order, spop, n, cum);
    else band_feature_kernel<1, ROWS, COLS, BANDS><<<grid, 256, 0, st>>>(prm, cs, w, order, spop, n, cum);
}

cudaError_t clear_counters(const BandWs &w, cudaStream_t st) {
    return cudaMemsetAsync(w.seen, 0, (size_t)(reinterpret_cast<char *>(w.seg) - reinterpret_cast<char *>(w.seen)), st);
}

}  // namespace

// 256x256 and 512x512 px (at smaller sizes G3 decides few pairs)
static bool size_covered(const Geo &g) { return g.N == 256 || g.N == 512; }

// the self-join: from 2,048 clips on, below which the band join takes less
// than the extra launches
bool band_mma_covers(const Geo &g, uint32_t n) { return size_covered(g) && n >= 2048; }

size_t band_mma_workspace(const Geo &g, uint32_t n) {
    if (!band_mma_covers(g, n)) return 0;
    BandWs w;
    return band_layout(g, n, n, list_room(n, n, true), true, true, nullptr, w);
}

// Decides the whole band into out / count / local unless *overflow (device)
// ends up 1; the caller then runs the band join.  order, spop, cum: the area
// sort.  ws: band_mma_workspace bytes, 256-byte aligned.
cudaError_t launch_band_mma(const pcl_params &prm, const pcl_clipset &cs, const uint32_t *order, const uint32_t *spop,
                            const uint32_t *cum, void *ws, pcl_pair *out, uint64_t cap, unsigned long long *count,
                            unsigned long long *local, const unsigned int **overflow, int num_sms,
                            unsigned long long wait_ns, cudaStream_t st) {
    const Geo g = make_geo(prm);
    const uint32_t n = cs.n_clips;
    BandWs w;
    band_layout(g, n, n, list_room(n, n, true), true, true, static_cast<char *>(ws), w);
    w.row_order = w.col_order = order;
    w.row_pop = w.col_pop = spop;
    *overflow = w.overflow;
    const cudaError_t e = clear_counters(w, st);
    if (e != cudaSuccess) return e;
    features<true, true, true>(prm, g, cs, w, order, spop, n, cum, st);
    if (g.N == 256)
        return launch_t<1024, 8, false>(prm, g, cs, cs, w, out, cap, count, local, num_sms, wait_ns, st);
    return launch_t<1024, 16, false>(prm, g, cs, cs, w, out, cap, count, local, num_sms, wait_ns, st);
}

// ---- two sets: the members' vectors apart (a served library keeps them), 256-byte aligned
size_t band_lib_bytes(const Geo &g, uint32_t n_lib) {
    if (!size_covered(g) || n_lib < 2048) return 0;
    const size_t blocks = (n_lib + kBlock - 1) / kBlock;
    return up(4 * kBlock * blocks) + blocks * kBlock * (size_t)kbytes_of(g.nb * g.nb);
}
static void lib_parts(void *lib, uint32_t n_lib, BandWs &w) {
    w.cb = static_cast<float *>(lib);
    w.Q = static_cast<unsigned char *>(lib) + up(4 * kBlock * (size_t)((n_lib + kBlock - 1) / kBlock));
}
cudaError_t launch_band_lib(const pcl_params &prm, const pcl_clipset &L, const uint32_t *order, const uint32_t *spop,
                            void *lib, cudaStream_t st) {
    const Geo g = make_geo(prm);
    BandWs w;
    band_layout(g, 0, L.n_clips, 0, false, false, nullptr, w);
    lib_parts(lib, L.n_clips, w);
    features<false, true, false>(prm, g, L, w, order, spop, L.n_clips, nullptr, st);
    return cudaGetLastError();
}

// the most queries whose list fits; more of them take the band join
uint32_t band_cross_most(uint32_t n_lib) { return (uint32_t)(kMaxList / ((uint64_t)n_lib / 256 + 64)); }

// 0: not covered
size_t band_cross_workspace(const Geo &g, uint32_t nq, uint32_t n_lib) {
    if (nq > band_cross_most(n_lib)) return 0;
    BandWs w;
    return band_layout(g, nq, n_lib, list_room(nq, n_lib, false), false, false, nullptr, w);
}

// as launch_band_mma for the queries Q (area order qorder, qspop; bands beg,
// end in the library's area order) against the library with its vectors lib
cudaError_t launch_band_cross(const pcl_params &prm, const pcl_clipset &Q, const pcl_clipset &L,
                              const uint32_t *lib_order, const uint32_t *lib_spop, void *lib, const uint32_t *qorder,
                              const uint32_t *qspop, uint32_t *beg, uint32_t *end, void *ws, pcl_pair *out,
                              uint64_t cap, unsigned long long *count, unsigned long long *local,
                              const unsigned int **overflow, int num_sms, unsigned long long wait_ns, cudaStream_t st) {
    const Geo g = make_geo(prm);
    BandWs w;
    band_layout(g, Q.n_clips, L.n_clips, list_room(Q.n_clips, L.n_clips, false), false, false, static_cast<char *>(ws), w);
    lib_parts(lib, L.n_clips, w);
    w.beg = beg;
    w.end = end;
    w.row_order = qorder;
    w.row_pop = qspop;
    w.col_order = lib_order;
    w.col_pop = lib_spop;
    *overflow = w.overflow;
    const cudaError_t e = clear_counters(w, st);
    if (e != cudaSuccess) return e;
    features<true, false, false>(prm, g, Q, w, qorder, qspop, Q.n_clips, nullptr, st);
    if (g.N == 256)
        return launch_t<1024, 8, true>(prm, g, Q, L, w, out, cap, count, local, num_sms, wait_ns, st);
    return launch_t<1024, 16, true>(prm, g, Q, L, w, out, cap, count, local, num_sms, wait_ns, st);
}

}  // namespace pcl
