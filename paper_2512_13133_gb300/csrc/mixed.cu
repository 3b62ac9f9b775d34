// a9: a mixed batch -- pairs of several raster size classes, cosine (FFT phase
// correlation) and edge (Min-Max) modes together, with uneven candidate lists.
//
// The work list holds the cosine items first, then the edge items.  Every
// kernel is persistent (a grid sized to the GPU) and finds its items in the
// list itself, so the whole batch is a fixed sequence of launches that a CUDA
// graph can replay: the edge items (edge_records, as for a pair list); the cosine gates, at full occupancy (the alignment
// bodies' registers and shared memory would leave ten warps per SM); then per
// size class the alignment of the items the gates left, marked in their
// records, by the FFT body of that size (512x512 px, beyond its shared memory:
// the exact window scan).  The register DFT radix (2 or 4), the CTAs per SM and
// the items a gating warp claims are tuning parameters (chosen by the
// autotuner).  5.2 M items over 4 x 5,000 clips of 64-512 px: 2.34 ms against
// 7.7 with gates, alignment and edge items in one kernel of 320-thread CTAs.
#include "edge_dev.cuh"
#include "exact_dev.cuh"
#include "fft_dev.cuh"
#include "rect_corr.cuh"

namespace pcl {

namespace {

using namespace fft_dev;
using namespace exact_dev;
using namespace edge_dev;

constexpr int kMaxClasses = 4;
constexpr int kClaimMax = 64;         // cosine items a warp claims at a time, at most (a tuning parameter)
constexpr uint16_t kPending = rect_corr::kRectPending;  // flags of a record whose item still needs its alignment

struct MixedArgs {
    pcl_params prm[kMaxClasses];
    pcl_clipset cs[kMaxClasses];
    uint32_t n_classes;
};

__global__ void mark_mixed_kernel(MixedArgs args, const pcl_work *work, uint64_t n_cos) {
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_cos;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const pcl_work w = work[t];
        if (w.cls >= args.n_classes) continue;
        const pcl_clipset &c = args.cs[w.cls];
        if (!c.spec_state || make_geo(args.prm[w.cls]).P > 32) continue;
        if (w.a < c.n_clips && c.spec_state[w.a] == 0) c.spec_state[w.a] = 2;
        if (w.b < c.n_clips && c.spec_state[w.b] == 0) c.spec_state[w.b] = 2;
    }
}

// Cosine items, `claim` consecutive ones per warp at a time.  A lane takes an
// item's indices, emptiness and areas (G1, which ends most items of unrelated
// clips) and the largest overlap that fails Eq. 2; the warp then takes G3 and G2 of the rest
// one after the other, the next item's first 64 blocks loading while one is
// tested.  An item that ends here gets its record, the others a record with
// flags = kPending.  Bound by issue slots: 2.6 M items, 1,090 us against 1,400 with the
// class's geometry, the overlap bound and the areas found by the whole warp for each item.
__global__ void __launch_bounds__(256) mixed_gate_kernel(MixedArgs args, const pcl_work *work, uint64_t n_cos,
                                                         pcl_record *out, unsigned long long *cursor, int claim) {
    const unsigned full = 0xffffffffu;
    __shared__ uint16_t g2_scratch[8 * kG2Scratch];
    __shared__ Geo geo[kMaxClasses];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t *scratch = g2_scratch + warp * kG2Scratch;
    if (threadIdx.x < args.n_classes) geo[threadIdx.x] = make_geo(args.prm[threadIdx.x]);
    __syncthreads();
    for (;;) {
        uint64_t t0 = 0;
        if (lane == 0) t0 = atomicAdd(cursor, (unsigned long long)claim);
        t0 = __shfl_sync(full, t0, 0);
        if (t0 >= n_cos) break;
        const uint64_t t1 = min(n_cos, t0 + (uint64_t)claim);
        for (uint64_t b = t0; b < t1; b += 32) {
            const uint64_t t = b + lane;
            pcl_work w{};
            int um = 0, area_a = 0, area_b = 0;
            bool open = false;
            pcl_record rec{};
            if (t < t1) {
                w = work[t];
                rec.a = w.a;
                rec.b = w.b;
                rec.mode = PCL_MODE_COSINE;
                if (w.cls >= args.n_classes || w.a >= args.cs[w.cls].n_clips || w.b >= args.cs[w.cls].n_clips) {
                    rec.flags = PCL_GATE_BAD_INDEX;
                } else {
                    const pcl_params &prm = args.prm[w.cls];
                    const pcl_clipset &cs = args.cs[w.cls];
                    const Geo &g = geo[w.cls];
                    const uint64_t pa = cs.pop[w.a], pb = cs.pop[w.b];
                    const uint64_t mn = pa < pb ? pa : pb, mx = pa < pb ? pb : pa;
                    if ((g.P > 32 && (g.P != 64 || prm.shift_rule != PCL_SHIFT_EXACT_ARGMAX)) || g.S > g.N / 16) {
                        rec.flags = PCL_GATE_UNSUPPORTED;
                    } else if (mx == 0) {
                        rec.flags = PCL_F_EMPTY;
                        rec.sim = 1.0f;
                        rec.pass = 1;
                    } else if (prm.flags & PCL_P_NO_GATES) {
                        rec.flags = kPending;
                    } else if (!((uint64_t)prm.cos_den * prm.cos_den * mn > (uint64_t)prm.cos_num * prm.cos_num * mx)) {
                        rec.flags = PCL_GATE_G1_AREA;
                    } else {
                        open = true;
                        area_a = (int)pa;
                        area_b = (int)pb;
                        um = (int)cos_umax(pa, pb, prm.cos_num, prm.cos_den);
                    }
                }
            }
            unsigned m = __ballot_sync(full, open);
            uint32_t ca = 0, da = 0, cb = 0, db = 0;  // the next item's first chunk: counts and neighbourhood sums
            auto fetch = [&](int q) {
                const uint32_t c = __shfl_sync(full, (uint32_t)w.cls, q);
                const uint32_t qa = __shfl_sync(full, w.a, q), qb = __shfl_sync(full, w.b, q);
                const int nb2 = geo[c].nb * geo[c].nb, words = nb2 / 2;
                const uint32_t *x = reinterpret_cast<const uint32_t *>(args.cs[c].blk) + (size_t)qa * nb2;
                const uint32_t *y = reinterpret_cast<const uint32_t *>(args.cs[c].blk) + (size_t)qb * nb2;
                const bool v = lane < words;
                ca = v ? __ldg(x + lane) : 0u;
                da = v ? __ldg(x + words + lane) : 0u;
                cb = v ? __ldg(y + lane) : 0u;
                db = v ? __ldg(y + words + lane) : 0u;
            };
            if (m) fetch(__ffs(m) - 1);
            while (m) {
                const int q = __ffs(m) - 1;
                m &= m - 1u;
                const uint32_t c = __shfl_sync(full, (uint32_t)w.cls, q);
                const uint32_t qa = __shfl_sync(full, w.a, q), qb = __shfl_sync(full, w.b, q);
                const int u = __shfl_sync(full, um, q);
                const int tA = __shfl_sync(full, area_a, q) - u, tB = __shfl_sync(full, area_b, q) - u;
                // G3 (warp_g3_rejects), 64 blocks at a time
                uint32_t sa = __reduce_add_sync(full, ca - __vminu2(ca, db));
                uint32_t sb = __reduce_add_sync(full, cb - __vminu2(cb, da));
                if (m) fetch(__ffs(m) - 1);
                int DA = (int)((sa & 0xffffu) + (sa >> 16)), DB = (int)((sb & 0xffffu) + (sb >> 16));
                bool rej = DA >= tA || DB >= tB;
                const Geo &g = geo[c];
                const pcl_clipset &cs = args.cs[c];
                const int nb2 = g.nb * g.nb, words = nb2 / 2;
                const uint32_t *x = reinterpret_cast<const uint32_t *>(cs.blk) + (size_t)qa * nb2;
                const uint32_t *y = reinterpret_cast<const uint32_t *>(cs.blk) + (size_t)qb * nb2;
                for (int k = 32 + lane; !rej && k < words; k += 32) {  // past 32 words there are a multiple of 32
                    const uint32_t c0 = __ldg(x + k), d0 = __ldg(x + words + k), c1 = __ldg(y + k),
                                   d1 = __ldg(y + words + k);
                    sa = __reduce_add_sync(full, c0 - __vminu2(c0, d1));
                    sb = __reduce_add_sync(full, c1 - __vminu2(c1, d0));
                    DA += (int)((sa & 0xffffu) + (sa >> 16));
                    DB += (int)((sb & 0xffffu) + (sb >> 16));
                    rej = DA >= tA || DB >= tB;
                }
                uint16_t flags = PCL_GATE_G3_DENSITY;
                if (!rej) {
                    const uint16_t *pa = cs.prof + (size_t)qa * 2 * g.N, *pb = cs.prof + (size_t)qb * 2 * g.N;
                    bool g2;
                    switch (g.N) {
                        case 64: g2 = warp_g2_rejects_groups<2>(pa, pb, g.S, u, lane, scratch); break;
                        case 128: g2 = warp_g2_rejects_groups<4>(pa, pb, g.S, u, lane, scratch); break;
                        case 256: g2 = warp_g2_rejects_groups<8>(pa, pb, g.S, u, lane, scratch); break;
                        default: g2 = warp_g2_rejects_groups<16>(pa, pb, g.S, u, lane, scratch); break;
                    }
                    flags = g2 ? PCL_GATE_G2_PROFILE : kPending;
                }
                if (lane == q) rec.flags = flags;
            }
            if (t < t1) out[t] = rec;
        }
    }
}

// The pending items of a 512x512 px class c from their rectangles
// (rect_corr.cuh), a warp per item; those it cannot take stay pending.
constexpr int kRectWarps = 4;

__global__ void __launch_bounds__(32 * kRectWarps) mixed_rect_kernel(pcl_params prm, pcl_clipset cs, uint32_t c,
                                                                     const pcl_work *work, uint64_t n_cos,
                                                                     pcl_record *out) {
    extern __shared__ __align__(16) unsigned char mixed_sm[];
    const Geo g = make_geo(prm);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int psh = (g.p & (g.p - 1)) == 0 ? 31 - __clz(g.p) : -1;
    const rect_corr::Scratch s = rect_corr::scratch_at(mixed_sm + warp * rect_corr::scratch_bytes(g.S), g.S);
    const uint64_t gw = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t base = 32 * gw; base < n_cos; base += 32 * nw) {
        const uint64_t t = base + lane;
        unsigned m = __ballot_sync(0xffffffffu, t < n_cos && out[t].flags == kPending && work[t].cls == c);
        while (m) {
            const int src = __ffs(m) - 1;
            m &= m - 1u;
            const pcl_pair pr{work[base + src].a, work[base + src].b};
            if (cs.pop[pr.a] != 0 && cs.pop[pr.b] != 0)
                rect_corr::rect_record(prm, g, psh, cs, cs, pr, s, -1, out + base + src, lane);
        }
    }
}

// The pending items of class c, aligned one at a time by a whole CTA with the
// engine of the class's size (P = N / 8; 64: the exact scan of 512^2 px).  A
// CTA claims up to kScan items and collects the pending ones of its class.  Of a list
// cut into C claims, claim c holds the groups of 32 consecutive items c, c + C, ..:
// pending items lie side by side (one clip's, one class's), and a claim of 512
// consecutive ones left them to a few CTAs (2,048 side by side: 12.8 ms, now 0.95, at 256x256
// px, 8.3 and 0.73 at 512x512).  A claim is an eighth of a
// CTA's share at most, so that short lists reach every CTA.
constexpr int kScan = 512;

template <int P>
struct AlignCta {
    static constexpr int threads = P == 64 ? exact_threads<8>() : 32 * 2 * ((9 * P / 2 + 1 + 31) / 32);
    static constexpr int ctas = P == 64 || P == 16 ? 2 : P == 32 ? 1 : 4;  // resident per SM
    static constexpr size_t smem() {
        if constexpr (P == 64) return exact_smem<8, 32>();
        else return PairSmem<P>::bytes;
    }
};

template <int P, int RADIX>
__global__ void __launch_bounds__(AlignCta<P>::threads, AlignCta<P>::ctas)
    mixed_align_kernel(pcl_params prm, pcl_clipset cs, uint32_t c, const pcl_work *work, uint64_t n_cos,
                       pcl_record *out, unsigned long long *cursor) {
    __shared__ uint16_t list[kScan];
    __shared__ int count;
    __shared__ unsigned long long at;
    if constexpr (P != 64) load_pair_table<P>();
    const uint64_t groups = (n_cos + 31) / 32, share = groups / (8 * (uint64_t)gridDim.x);
    const uint32_t per = share < 1 ? 1u : share < kScan / 32 ? (uint32_t)share : kScan / 32;  // groups a claim
    const uint64_t claims = (groups + per - 1) / per;
    auto item = [&](uint64_t c, uint32_t k) { return 32 * (c + (k >> 5) * claims) + (k & 31u); };
    for (;;) {
        __syncthreads();  // the previous list is no longer read
        if (threadIdx.x == 0) {
            count = 0;
            at = atomicAdd(cursor, 1ull);
        }
        __syncthreads();
        const uint64_t claim = at;
        if (claim >= claims) break;
        for (uint32_t k = threadIdx.x; k < 32 * per; k += blockDim.x) {
            const uint64_t t = item(claim, k);
            if (t < n_cos && out[t].flags == kPending && work[t].cls == c) list[atomicAdd(&count, 1)] = (uint16_t)k;
        }
        __syncthreads();
        const int n = count;
        for (int k = 0; k < n; ++k) {
            const uint64_t t = item(claim, list[k]);
            const pcl_pair pr{work[t].a, work[t].b};
            if constexpr (P == 64) exact_body<8, 32>(prm, cs, cs, pr, out + t);
            else pair_body<P, RADIX>(prm, cs, cs, pr, out + t, true);
            __syncthreads();
        }
    }
}

// Edge items (edge_records)
struct EdgeItems {
    static constexpr bool one_class = false;
    MixedArgs args;
    const pcl_work *work;
    __device__ __forceinline__ bool item(uint64_t t, pcl_pair &pr, uint32_t &cls) const {
        const pcl_work w = work[t];
        pr = pcl_pair{w.a, w.b};
        cls = w.cls < args.n_classes ? w.cls : 0u;
        return w.cls < args.n_classes && w.a < args.cs[cls].n_clips && w.b < args.cs[cls].n_clips;
    }
    __device__ __forceinline__ const pcl_params &params(uint32_t c) const { return args.prm[c]; }
    __device__ __forceinline__ const pcl_clipset &A(uint32_t c) const { return args.cs[c]; }
    __device__ __forceinline__ const pcl_clipset &B(uint32_t c) const { return args.cs[c]; }
};

__global__ void __launch_bounds__(256, 3) mixed_edge_kernel(EdgeItems items, uint64_t n, pcl_record *out) {
    edge_records(items, n, out);
}

template <int P, int RADIX>
cudaError_t align_t(const pcl_params &prm, const pcl_clipset &cs, uint32_t c, const pcl_work *work, uint64_t n_cos,
                    pcl_record *out, unsigned long long *cursor, uint32_t ctas_per_sm, int num_sms, cudaStream_t st) {
    const size_t sm = AlignCta<P>::smem();
    auto *kern = mixed_align_kernel<P, RADIX>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, AlignCta<P>::threads, sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    if (ctas_per_sm != 0 && (int)ctas_per_sm < per_sm) per_sm = (int)ctas_per_sm;
    kern<<<(unsigned)(num_sms * per_sm), AlignCta<P>::threads, sm, st>>>(prm, cs, c, work, n_cos, out, cursor);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_spectra(const pcl_params &, const pcl_clipset &, const uint32_t *, uint32_t, bool, cudaStream_t);

cudaError_t launch_mixed(const pcl_params *prm, const pcl_clipset *sets, uint32_t n_classes, const pcl_work *work,
                         uint64_t n_cos, uint64_t n, pcl_record *out, unsigned long long *cursor, uint32_t radix,
                         uint32_t ctas_per_sm, uint32_t items_per_warp, int num_sms, cudaStream_t st) {
    if (n_classes == 0 || n_classes > kMaxClasses) return cudaErrorInvalidValue;
    const int claim = items_per_warp == 0 ? 16 : (int)items_per_warp;
    if (claim > kClaimMax) return cudaErrorInvalidValue;
    MixedArgs args{};
    args.n_classes = n_classes;
    for (uint32_t c = 0; c < n_classes; ++c) {
        args.prm[c] = prm[c];
        args.cs[c] = sets[c];
    }
    cudaError_t e = cudaMemsetAsync(cursor, 0, sizeof(unsigned long long) * (1 + kMaxClasses), st);
    if (e != cudaSuccess) return e;
    if (n_cos) {
        mark_mixed_kernel<<<1024, 256, 0, st>>>(args, work, n_cos);
        for (uint32_t c = 0; c < n_classes; ++c) {
            if (!sets[c].spec_state || make_geo(prm[c]).P > 32) continue;
            if ((e = launch_spectra(prm[c], sets[c], nullptr, 0, true, st)) != cudaSuccess) return e;
        }
    }
    if (n == 0) return cudaSuccess;
    if (n > n_cos) mixed_edge_kernel<<<num_sms * 3, 256, 0, st>>>(EdgeItems{args, work + n_cos}, n - n_cos, out + n_cos);
    if (n_cos) {
        mixed_gate_kernel<<<num_sms * 8, 256, 0, st>>>(args, work, n_cos, out, cursor, claim);
        for (uint32_t c = 0; c < n_classes; ++c) {
            const Geo g = make_geo(prm[c]);
            // no item is pending past this marker (PCL_GATE_UNSUPPORTED), and at 512x512 px
            // the tables of shifts would outgrow shared memory from S = 60 on
            if (g.S > g.N / 16) continue;
            unsigned long long *cur = cursor + 1 + c;
            switch (g.P * 2 + (radix == 4 ? 1 : 0)) {
                case 16: e = align_t<8, 2>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st); break;
                case 17: e = align_t<8, 4>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st); break;
                case 32: e = align_t<16, 2>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st); break;
                case 33: e = align_t<16, 4>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st); break;
                case 64: e = align_t<32, 2>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st); break;
                case 65: e = align_t<32, 4>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st); break;
                default: {
                    const size_t rs = kRectWarps * rect_corr::scratch_bytes(g.S);
                    e = cudaFuncSetAttribute(mixed_rect_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rs);
                    if (e != cudaSuccess) return e;
                    mixed_rect_kernel<<<num_sms * 3, 32 * kRectWarps, rs, st>>>(prm[c], sets[c], c, work, n_cos, out);
                    e = align_t<64, 2>(prm[c], sets[c], c, work, n_cos, out, cur, ctas_per_sm, num_sms, st);
                    break;
                }
            }
            if (e != cudaSuccess) return e;
        }
    }
    return cudaGetLastError();
}

}  // namespace pcl
