// a3-a6: FFT phase correlation (Sec. 3.2.1, Eqs. 3-5) and the cosine test at
// the optimal shift (Sec. 2.2.1, Eq. 2).
//
// FFT side L = 9P with P = N/8 a power of two: every shift |s| <= N/8 of the
// zero-padded linear correlation is alias-free (L >= N + S).  All transforms
// use one decomposition, index = 9*i1 + i2 on the input side and
// k = k1 + P*k2 on the output side:
//   X[k1 + P k2] = sum_i2 w9^(k2 i2) wL^(k1 i2) sum_i1 x[9 i1 + i2] wP^(k1 i1)
// i.e. nine P-point DFTs in registers (radix-2, compile-time twiddles), a
// twiddle, and P nine-point DFTs (3 x 3).
//
// Forward (per clip, cached): R2C of the raster zero-padded to L x L.  Rows
// are transformed two at a time as one complex sequence and split; then the
// L/2+1 columns.  The spectrum is stored [ky][kx] with kx contiguous.
//
// Per pair (one CTA): C = F_A conj(F_B) on the half spectrum; the phase-
// correlation spectrum R = C/|C| (Eq. 4; bins with |C| <= 1e-6 |A||B| set to
// 0, |A||B| = C(0) being the largest |C|).  Inverse pass 1 runs along ky for
// every kx column, pruned to the 2*(P/2)+1 output rows |dy| <= P/2: with
// outputs n = n1 + P n2 only n2 = 0 (dy >= 0) and n2 = 8 (dy < 0) are kept,
// so the nine-point stage collapses to one twiddled sum per output.  Pass 2
// packs the two Hermitian rows as R + iC into one complex sequence over kx
// and gives r_pcm(s) (real part) and c(s) (imaginary part), again pruned.
// The correlation is rounded to integers; the residual guard (any window
// entry more than 0.25 from an integer) and a popcount check of c at the
// chosen shift fall back to an exact popcount scan of the whole window.
#include <climits>

#include "exact_dev.cuh"
#include "rect_corr.cuh"
#include "fft_dev.cuh"

namespace pcl {

cudaError_t launch_rect_pairs(const pcl_params &, const pcl_clipset &, const pcl_clipset &, const pcl_pair *, uint64_t,
                              const unsigned long long *, pcl_record *, uint32_t *, int, unsigned long long *,
                              cudaStream_t);

namespace {

using namespace fft_dev;
using namespace exact_dev;

// ---------------------------------------------------------------- forward
// One CTA per clip.  Rows are transformed two at a time (2t, 2t + 1) as one
// complex sequence; in a raster of rectangles many consecutive row pairs are
// equal (a clip of 21 rectangles has about 55 runs of equal pairs among its
// 128), and equal pairs have equal transforms, so each run is transformed once:
// its rows go to rows 2u, 2u + 1 of the clip's spectrum buffer, and the column
// pass reads row y of the raster from its run's row (mostly from L1).  288
// threads = 9 warps: one P-point DFT task each (32 sequences x 9).  Bound by
// issue slots and L2 traffic; 4,096 clips of 256x256 px: 745 us against 1,400 with
// every row pair transformed, 256 threads and twiddles by double sincospi in every CTA.
constexpr int kSpecThreads = 288;

template <int P>
__global__ void __launch_bounds__(kSpecThreads, 2) spectra_kernel(pcl_params prm, pcl_clipset cs,
                                                                  const uint32_t *list, uint32_t n_list,
                                                                  uint8_t want_state) {
    constexpr int L = 9 * P, N = 8 * P, NW = N / 64, LH = L / 2 + 1;
    constexpr int LS = (LH + 3) & ~3;
    constexpr int CH = 32;  // row pairs or columns per chunk
    uint32_t c;
    if (list) {
        if (blockIdx.x >= n_list) return;
        c = list[blockIdx.x];
    } else {
        c = blockIdx.x;
        if (c >= cs.n_clips) return;
        if (cs.spec_state[c] != want_state && !(want_state == 0 && cs.spec_state[c] == 2)) return;
    }
    extern __shared__ __align__(16) unsigned char smem[];
    float2 *tw = reinterpret_cast<float2 *>(smem);                 // L
    uint64_t *bits = reinterpret_cast<uint64_t *>(tw + L);          // N * NW
    float2 *vb = reinterpret_cast<float2 *>(bits + N * NW);         // CH * 9 * (P + 1)
    __shared__ uint16_t row_at[N];      // row of the buffer holding raster row y's transform
    __shared__ uint8_t run_first[N / 2];  // first row pair of each run
    __shared__ uint32_t warp_runs[4];
    load_twiddles<L>(tw, -1);
    const uint64_t *src = cs.bits + (size_t)c * N * NW;
    for (int t = threadIdx.x; t < N * NW; t += blockDim.x) bits[t] = src[t];
    float2 *spec = reinterpret_cast<float2 *>(cs.spec) + (size_t)c * L * LS;
    __syncthreads();
    // runs of equal row pairs
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned starts = 0u;
    if (threadIdx.x < N / 2) {
        const int t = threadIdx.x;
        bool start = t == 0;
#pragma unroll
        for (int w = 0; w < 2 * NW; ++w) start = start || bits[2 * t * NW + w] != bits[2 * (t - 1) * NW + w];
        starts = __ballot_sync(0xffffffffu, start);
        if (lane == 0) warp_runs[warp] = (uint32_t)__popc(starts);
    }
    __syncthreads();
    int runs = 0;
#pragma unroll
    for (int w = 0; w < (N / 2) / 32; ++w) runs += (int)warp_runs[w];
    if (threadIdx.x < N / 2) {
        int u = __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
        for (int w = 0; w < warp; ++w) u += (int)warp_runs[w];
        const int t = threadIdx.x;
        row_at[2 * t] = (uint16_t)(2 * u);
        row_at[2 * t + 1] = (uint16_t)(2 * u + 1);
        if ((starts >> lane) & 1u) run_first[u] = (uint8_t)t;
    }
    __syncthreads();

    // ---- rows: the runs' pairs (2t, 2t+1) as one complex sequence
    for (int u0 = 0; u0 < runs; u0 += CH) {
        const int cnt = min(CH, runs - u0);
        for (int task = threadIdx.x; task < CH * 9; task += blockDim.x) {
            const int tl = task % CH, i2 = task / CH;
            if (tl >= cnt) continue;
            const int t = run_first[u0 + tl];
            float2 v[P];
#pragma unroll
            for (int i1 = 0; i1 < P; ++i1) {
                const int x = 9 * i1 + i2;
                v[i1] = (x < N) ? make_float2(bitf(bits, NW, 2 * t, x), bitf(bits, NW, 2 * t + 1, x))
                                : make_float2(0.f, 0.f);
            }
            dft_pow2<P, -1>(v);
#pragma unroll
            for (int k1 = 0; k1 < P; ++k1) vb[vslot<P>(tl, i2, k1)] = v[k1];
        }
        __syncthreads();
        for (int task = threadIdx.x; task < cnt * P; task += blockDim.x) {
            const int k1 = task % P, tl = task / P;
            float2 u[9];
#pragma unroll
            for (int i2 = 0; i2 < 9; ++i2) u[i2] = cmul(vb[vslot<P>(tl, i2, k1)], tw[(k1 * i2) % L]);
            dft9<-1>(u);
#pragma unroll
            for (int k2 = 0; k2 < 9; ++k2) vb[vslot<P>(tl, k2, k1)] = u[k2];
        }
        __syncthreads();
        for (int task = threadIdx.x; task < cnt * LH; task += blockDim.x) {
            const int kx = task % LH, tl = task / LH;
            const int km = (L - kx) % L;
            const float2 xk = vb[vslot<P>(tl, kx / P, kx % P)];
            const float2 xm = cconj(vb[vslot<P>(tl, km / P, km % P)]);
            const float2 fe = cscale(cadd(xk, xm), 0.5f);
            const float2 d = csub(xk, xm);
            const float2 fo = make_float2(0.5f * d.y, -0.5f * d.x);  // d / (2i)
            spec[(size_t)(2 * (u0 + tl)) * LS + kx] = fe;
            spec[(size_t)(2 * (u0 + tl) + 1) * LS + kx] = fo;
        }
        __syncthreads();
    }
    // ---- columns kx in chunks of CH
    for (int c0 = 0; c0 < LH; c0 += CH) {
        for (int task = threadIdx.x; task < CH * 9; task += blockDim.x) {
            const int cl = task % CH, i2 = task / CH, kx = c0 + cl;
            float2 v[P];
#pragma unroll
            for (int i1 = 0; i1 < P; ++i1) {
                const int y = 9 * i1 + i2;
                v[i1] = (y < N && kx < LH) ? spec[(size_t)row_at[y < N ? y : 0] * LS + kx] : make_float2(0.f, 0.f);
            }
            dft_pow2<P, -1>(v);
#pragma unroll
            for (int k1 = 0; k1 < P; ++k1) vb[vslot<P>(cl, i2, k1)] = v[k1];
        }
        __syncthreads();
        for (int task = threadIdx.x; task < CH * P; task += blockDim.x) {
            const int cl = task % CH, k1 = task / CH, kx = c0 + cl;
            if (kx >= LH) continue;
            float2 u[9];
#pragma unroll
            for (int i2 = 0; i2 < 9; ++i2) u[i2] = cmul(vb[vslot<P>(cl, i2, k1)], tw[(k1 * i2) % L]);
            dft9<-1>(u);
#pragma unroll
            for (int k2 = 0; k2 < 9; ++k2) spec[(size_t)(k1 + P * k2) * LS + kx] = u[k2];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) cs.spec_state[c] = 1;
}

// mark clips referenced by a pair list whose spectrum is missing (state 2)
__global__ void mark_kernel(const pcl_pair *pairs, uint64_t n, const unsigned long long *d_n, uint8_t *state_a,
                            uint8_t *state_b, uint32_t na, uint32_t nb) {
    if (d_n && *d_n < n) n = *d_n;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const pcl_pair p = pairs[t];
        if (p.a < na && state_a[p.a] == 0) state_a[p.a] = 2;
        if (p.b < nb && state_b[p.b] == 0) state_b[p.b] = 2;
    }
}

// persistent: each CTA walks the pair list with a grid stride.  One CTA of ten
// warps per SM at P = 32 (registers and shared memory allow no second), so it is
// bound by latency: issue slots were half busy, a third of pass 1 was the wait
// for a step's 2 P loads and another third the sums in shared memory.  40,000 pairs of
// 256x256 px 8.73 -> 7.30 ms: the sums' next batch loading during an addition
// and the tables once per CTA 0.8 ms, the next step's rows and the rasters of
// the final check fetched into L2 0.6 ms, the order of the units over the schedulers
// 0.1 ms.  Measured on the way: pass 1's twiddles in shared memory instead of
// constant memory 10.0 ms, the leftover columns' halves sharing a warp 8.9 ms, the
// next pair's first rows fetched as well 8.1 ms.
template <int P>
__global__ void __launch_bounds__(32 * 2 * ((9 * P / 2 + 1 + 31) / 32), P == 32 ? 1 : P == 16 ? 2 : 4)
    pair_fft_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B, const pcl_pair *pairs, uint64_t npairs,
                    const unsigned long long *d_n, pcl_record *out) {
    if (d_n && *d_n < npairs) npairs = *d_n;
    load_pair_table<P>();
    for (uint64_t pid = blockIdx.x; pid < npairs; pid += gridDim.x) {
        __syncthreads();
        pair_body<P>(prm, A, B, pairs[pid], out + pid);
    }
}

// The exact window scan: at 512² the FFT body's buffers exceed shared memory,
// and at 128² / 256² it is the exact-scan engine.  rect_pair_kernel comes first
// (indices, emptiness, gates, and the record from the rectangles where it can);
// the pairs it leaves pending take the bound-pruned scan of the rasters
// (exact_body<NW, SMAX>, N = 64 NW, S <= SMAX = N/16), one pair per CTA
// iteration.  CTA b owns the pairs b, b + G, b + 2G, .. of a grid of G, looks at
// as many of them as it has threads and scans the pending ones: neighbours in
// a list mostly share a clip and are pending together, and consecutive
// pairs per CTA left most of the GPU idle (1,000 pairs of clips of 100 rectangles:
// 20.7 ms against 0.42 at 512x512 px, 2.65 against 0.09 at 256x256).  list (with its length n_list on the device): those pairs instead.
template <int NW, int SMAX>
__global__ void __launch_bounds__(exact_threads<NW>(), NW == 8 ? 2 : 6)
    exact_pair_kernel(pcl_params prm, pcl_clipset A, pcl_clipset B, const pcl_pair *pairs, uint64_t npairs,
                      const unsigned long long *d_n, pcl_record *out, unsigned long long *stats,
                      const uint32_t *list, const uint32_t *n_list) {
    if (list) {
        for (uint64_t k = blockIdx.x; k < *n_list; k += gridDim.x)
            exact_body<NW, SMAX>(prm, A, B, pairs[list[k]], out + list[k], stats);
        return;
    }
    constexpr int T = exact_threads<NW>();
    __shared__ uint16_t open_s[T];
    __shared__ int count;
    if (d_n && *d_n < npairs) npairs = *d_n;
    for (uint64_t t0 = blockIdx.x; t0 < npairs; t0 += (uint64_t)gridDim.x * T) {
        __syncthreads();  // the previous list is no longer read
        if (threadIdx.x == 0) count = 0;
        __syncthreads();
        const uint64_t t = t0 + (uint64_t)threadIdx.x * gridDim.x;
        if (t < npairs && out[t].flags == rect_corr::kRectPending) open_s[atomicAdd(&count, 1)] = (uint16_t)threadIdx.x;
        __syncthreads();
        const int n = count;
        for (int k = 0; k < n; ++k) {
            const uint64_t p = t0 + (uint64_t)open_s[k] * gridDim.x;
            exact_body<NW, SMAX>(prm, A, B, pairs[p], out + p, stats);
        }
    }
}

template <int P>
size_t spectra_smem() {
    constexpr int L = 9 * P, N = 8 * P;
    return sizeof(float2) * L + 8 * (size_t)N * (N / 64) + sizeof(float2) * 32 * 9 * (P + 1);
}

template <int P>
cudaError_t spectra_t(const pcl_params &prm, const pcl_clipset &cs, const uint32_t *list, uint32_t n_list,
                      uint8_t want, cudaStream_t st) {
    const size_t sm = spectra_smem<P>();
    cudaError_t e = cudaFuncSetAttribute(spectra_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const uint32_t grid = list ? n_list : cs.n_clips;
    if (grid == 0) return cudaSuccess;
    spectra_kernel<P><<<grid, kSpecThreads, sm, st>>>(prm, cs, list, n_list, want);
    return cudaGetLastError();
}

template <int P>
cudaError_t pair_t(const pcl_params &prm, const pcl_clipset &a, const pcl_clipset &b, const pcl_pair *pairs,
                   uint64_t n, const unsigned long long *d_n, pcl_record *out, int num_sms, cudaStream_t st) {
    const size_t sm = PairSmem<P>::bytes;
    cudaError_t e = cudaFuncSetAttribute(pair_fft_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    if (n == 0) return cudaSuccess;
    constexpr int LH = 9 * P / 2 + 1;
    const int threads = 32 * 2 * ((LH + 31) / 32);
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pair_fft_kernel<P>, threads, sm);
    if (e != cudaSuccess) return e;
    const uint64_t cap = (uint64_t)num_sms * (uint64_t)(per_sm > 0 ? per_sm : 1);
    const unsigned grid = (unsigned)(n < cap ? n : cap);
    pair_fft_kernel<P><<<grid, threads, sm, st>>>(prm, a, b, pairs, n, d_n, out);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_spectra(const pcl_params &prm, const pcl_clipset &cs, const uint32_t *list,
                           uint32_t n_list, bool requested_only, cudaStream_t st) {
    const Geo g = make_geo(prm);
    const uint8_t want = requested_only ? 2 : 0;
    switch (g.P) {
        case 8: return spectra_t<8>(prm, cs, list, n_list, want, st);
        case 16: return spectra_t<16>(prm, cs, list, n_list, want, st);
        case 32: return spectra_t<32>(prm, cs, list, n_list, want, st);
        default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_mark(const pcl_pair *pairs, uint64_t n, const unsigned long long *d_n, pcl_clipset &a,
                        pcl_clipset &b, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    mark_kernel<<<1024, 256, 0, st>>>(pairs, n, d_n, a.spec_state, b.spec_state, a.n_clips, b.n_clips);
    return cudaGetLastError();
}

template <int NW, int SMAX>
cudaError_t exact_t(const pcl_params &prm, const pcl_clipset &a, const pcl_clipset &b, const pcl_pair *pairs,
                    uint64_t n, const unsigned long long *d_n, pcl_record *out, int num_sms,
                    unsigned long long *stats, const uint32_t *list, const uint32_t *n_list, cudaStream_t st) {
    const size_t sm = exact_smem<NW, SMAX>();
    constexpr int kExactThreads = exact_threads<NW>();
    auto *kern = exact_pair_kernel<NW, SMAX>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess || n == 0) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kExactThreads, sm);
    if (e != cudaSuccess) return e;
    const uint64_t cap = (uint64_t)num_sms * (uint64_t)(per_sm > 0 ? per_sm : 1);
    const unsigned grid = (unsigned)(n < cap ? n : cap);
    kern<<<grid, kExactThreads, sm, st>>>(prm, a, b, pairs, n, d_n, out, stats, list, n_list);
    return cudaGetLastError();
}

cudaError_t launch_exact_pairs(const pcl_params &prm, const pcl_clipset &a, const pcl_clipset &b,
                               const pcl_pair *pairs, uint64_t n, const unsigned long long *d_n, pcl_record *out,
                               int num_sms, unsigned long long *stats, cudaStream_t st, const uint32_t *list,
                               const uint32_t *n_list) {
    const Geo g = make_geo(prm);
    if (g.S > g.N / 16) return cudaErrorNotSupported;
    if (!list) {
        const cudaError_t e = launch_rect_pairs(prm, a, b, pairs, n, d_n, out, nullptr, num_sms, stats, st);
        if (e != cudaSuccess) return e;
    }
    switch (g.N) {
        case 128: return exact_t<2, 8>(prm, a, b, pairs, n, d_n, out, num_sms, stats, list, n_list, st);
        case 256: return exact_t<4, 16>(prm, a, b, pairs, n, d_n, out, num_sms, stats, list, n_list, st);
        case 512: return exact_t<8, 32>(prm, a, b, pairs, n, d_n, out, num_sms, stats, list, n_list, st);
        default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_pair_fft(const pcl_params &prm, const pcl_clipset &a, const pcl_clipset &b,
                            const pcl_pair *pairs, uint64_t n, const unsigned long long *d_n, pcl_record *out,
                            int num_sms, cudaStream_t st) {
    const Geo g = make_geo(prm);
    switch (g.P) {
        case 8: return pair_t<8>(prm, a, b, pairs, n, d_n, out, num_sms, st);
        case 16: return pair_t<16>(prm, a, b, pairs, n, d_n, out, num_sms, st);
        case 32: return pair_t<32>(prm, a, b, pairs, n, d_n, out, num_sms, st);
        default: return cudaErrorNotSupported;
    }
}

}  // namespace pcl
