// a1: rasterisation of Manhattan clips and the per-clip signatures read by the
// lossless gates (Sec. 2.2.1 step 1; signatures for the pre-screening of
// Sec. 3.1 stage 1).
#include <climits>

#include "common.cuh"

namespace pcl {

namespace {

// grid cell of coordinate v (floor division, clamped to the 64 cells)
__device__ __forceinline__ int cell_of(int v, int csz) {
    const int q = v >= 0 ? v / csz : -((-v + csz - 1) / csz);
    return q < 0 ? 0 : (q > 63 ? 63 : q);
}

// first pixel index i (clamped to [0, N]) whose centre p i + p/2 is >= v:
// ceil((2 v - p) / (2 p)), the pixel-centre rule of a rectangle edge at v
__device__ __forceinline__ int pix_from(int v, long long p, int N) {
    const long long a = 2LL * v - p, b = 2 * p;
    long long q = a / b;
    if (a % b != 0 && a > 0) ++q;
    return (int)(q < 0 ? 0 : (q > N ? N : q));
}

// log2 of v when it is a power of two, else -1
__device__ __forceinline__ int log2_exact(int v) { return (v & (v - 1)) == 0 ? 31 - __clz(v) : -1; }

// pix_from with psh >= 0: the pitch is 1 << psh
__device__ __forceinline__ int pix_at(int v, int p, int psh, int N) {
    if (psh < 0) return pix_from(v, p, N);
    const long long q = (2LL * v + p - 1) >> (psh + 1);  // ceil((2 v - p) / (2 p))
    return (int)(q < 0 ? 0 : (q > N ? N : q));
}
// cell_of with csh >= 0: the cell side is 1 << csh
__device__ __forceinline__ int cell_at(int v, int csz, int csh) {
    return csh >= 0 ? min(max(v >> csh, 0), 63) : cell_of(v, csz);
}

template <int NW>
struct RasterCta {
    static constexpr int threads = NW == 8 ? 256 : 128;
    static constexpr int chunk = 128;  // rectangles staged at a time
    static constexpr int ctas = NW == 8 ? 4 : 12;  // resident per SM: registers and shared memory allow as many
};

// Indices of the nr rectangles by ascending area (ties by index) into order, by rank
// counting with all T threads of the CTA, the areas staged CHUNK at a time (5,000
// clips of 1,000 rectangles, 512x512 px: 10.1 ms by one warp from global memory, now
// 1.7).  Clips of more than CHUNK rectangles are rare.
template <int T, int CHUNK>
__device__ __forceinline__ void order_many(const int4 *r4, uint32_t nr, long long *areas, uint16_t *order) {
    auto area_of = [&](uint32_t m) {
        const int4 q = __ldg(r4 + m);
        return (long long)(q.z - q.x) * (long long)(q.w - q.y);
    };
    for (uint32_t t0 = 0; t0 < nr; t0 += T) {
        const uint32_t t = t0 + threadIdx.x;
        const long long at = t < nr ? area_of(t) : 0;
        uint32_t rank = 0;
        for (uint32_t base = 0; base < nr; base += CHUNK) {
            const uint32_t cnt = min((uint32_t)CHUNK, nr - base);
            __syncthreads();  // the areas staged before are no longer read
            for (uint32_t m = threadIdx.x; m < cnt; m += T) areas[m] = area_of(base + m);
            __syncthreads();
#pragma unroll 4
            for (uint32_t m = 0; m < cnt; ++m) rank += areas[m] < at + (base + m < t ? 1 : 0) ? 1u : 0u;
        }
        if (t < nr) order[rank] = (uint16_t)t;
    }
}

// One CTA per clip.  The rectangles (a chunk at a time) become pixel
// ranges in shared memory; then each warp has one job with a lane per
// rectangle: setting the rows' bits, adding the pixels of its 16x16 blocks and
// the ends of its column run to a difference array, marking the occupancy
// grid, ordering by area and the edge signature.  If the pixels of all ranges
// add up to the raster's ones, no two rectangles share a pixel and those sums
// are the block counts and (after a prefix sum) the column counts; otherwise
// both are counted from the rows.  Bound by issue slots and the latency of each
// warp's job; the output is written once, 16 bytes a thread.  100,000 clips of
// 256x256 px: 413 us (2.7 TB/s) against 1,265 us with a thread per row testing
// every rectangle and column counts by bit transposes; 12 CTAs per SM (40
// registers) against 10: 413 and 446 us.
template <int NW>
__global__ void __launch_bounds__(RasterCta<NW>::threads, RasterCta<NW>::ctas) raster_kernel(pcl_params prm, pcl_clipset cs) {
    constexpr int N = 64 * NW, W32 = 2 * NW, NB = 4 * NW, NB2 = NB * NB;
    constexpr int T = RasterCta<NW>::threads, CHUNK = RasterCta<NW>::chunk;
    constexpr int SR = W32 + 1;  // row stride in shared memory (odd: the lanes of a rectangle's rows spread over the banks)
    constexpr int FILL = T / 32 - 3;  // warps setting bits
    const Geo g = make_geo(prm);
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int4 rs[CHUNK];          // pixel ranges {i0, i1, j0, j1} of staged rectangles
    __shared__ int4 rq[CHUNK];          // the rectangles
    __shared__ long long areas[CHUNK];       // of the staged rectangles
    // zeroed together: the rows, ones entering (leaving) at each column, block
    // counts, and the occupancy grid's 64 rows (low and high word)
    constexpr int Z = (N * SR + (N + 4) + NB2 + 128 + 3) / 4;
    __shared__ uint4 zeroed[Z];
    uint32_t *rows = reinterpret_cast<uint32_t *>(zeroed);
    int *diff = reinterpret_cast<int *>(rows + N * SR);
    uint32_t *cnt_s = rows + N * SR + N + 4, *occ_s = cnt_s + NB2;
    __shared__ uint32_t red[T / 32];
    __shared__ unsigned long long area_sum;  // pixels of all ranges
    const uint32_t r0 = cs.rect_off[c], r1 = cs.rect_off[c + 1], nr = r1 - r0;
    const int4 *r4 = reinterpret_cast<const int4 *>(cs.rects) + r0;
    const int psh = log2_exact(g.p), csz = g.W / 64, csh = log2_exact(csz);
    for (int t = tid; t < Z; t += T) zeroed[t] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) area_sum = 0ull;
    // edge signature (warp 0): bbox over edges that are not on the window border
    int hasx = 0, hasy = 0, border = 0;
    int lox = INT_MAX, hix = INT_MIN, loy = INT_MAX, hiy = INT_MIN;
    for (uint32_t base = 0; base < nr; base += CHUNK) {
        const uint32_t cnt = min((uint32_t)CHUNK, nr - base);
        __syncthreads();
        // pixel (i, j) is set when x0 <= p i + p/2 < x1 and y0 <= p j + p/2 < y1
        // (doubled: 2 x0 <= 2 p i + p < 2 x1): columns [i0, i1), rows [j0, j1)
        for (uint32_t t = tid; t < cnt; t += T) {
            const int4 q = __ldg(r4 + base + t);
            rq[t] = q;
            areas[t] = (long long)(q.z - q.x) * (long long)(q.w - q.y);
            rs[t] = make_int4(pix_at(q.x, g.p, psh, N), pix_at(q.z, g.p, psh, N), pix_at(q.y, g.p, psh, N),
                              pix_at(q.w, g.p, psh, N));
        }
        __syncthreads();
        if (warp >= 3) {
            // bits: lane = rectangle; the warps share its rows
            for (uint32_t t = lane; t < cnt; t += 32) {
                const int4 q = rs[t];
                if (q.x >= q.y) continue;
                const int w0 = q.x >> 5, w1 = (q.y - 1) >> 5;
                const uint32_t first = 0xffffffffu << (q.x & 31), last = 0xffffffffu >> (31 - ((q.y - 1) & 31));
                for (int j = q.z + (warp - 3); j < q.w; j += FILL) {
                    uint32_t *row = rows + j * SR;
                    if (w0 == w1) {
                        atomicOr(row + w0, first & last);
                    } else {
                        atomicOr(row + w0, first);
                        for (int w = w0 + 1; w < w1; ++w) atomicOr(row + w, 0xffffffffu);
                        atomicOr(row + w1, last);
                    }
                }
            }
        } else if (warp == 2) {
            // block counts and column differences
            unsigned long long area = 0;
            for (uint32_t t = lane; t < cnt; t += 32) {
                const int4 q = rs[t];
                const int h = q.w - q.z;
                if (q.x >= q.y || h <= 0) continue;
                area += (unsigned long long)(q.y - q.x) * (unsigned)h;
                atomicAdd(diff + q.x, h);
                atomicAdd(diff + q.y, -h);
                for (int by = q.z >> 4; by <= (q.w - 1) >> 4; ++by) {
                    const int hh = min(q.w, 16 * by + 16) - max(q.z, 16 * by);
                    for (int bx = q.x >> 4; bx <= (q.y - 1) >> 4; ++bx)
                        atomicAdd(cnt_s + by * NB + bx, (uint32_t)(hh * (min(q.y, 16 * bx + 16) - max(q.x, 16 * bx))));
                }
            }
            for (int o = 16; o; o >>= 1) area += __shfl_xor_sync(0xffffffffu, area, o);
            if (lane == 0) area_sum += area;
        } else if (warp == 1) {
            // 64 x 64 occupancy grid (cell side W/64): a cell is marked when it holds an
            // integer point of some rectangle's interior, so two rectangles that
            // overlap with positive area always share a marked cell
            for (uint32_t t = lane; t < cnt; t += 32) {
                const int4 q = rq[t];
                if (q.z <= q.x || q.w <= q.y) continue;
                const int y0 = cell_at(q.y, csz, csh), y1 = cell_at(q.w - 1, csz, csh);
                const int x0 = cell_at(q.x, csz, csh), x1 = cell_at(q.z - 1, csz, csh);
                const unsigned long long m = (~0ull >> (63 - (x1 - x0))) << x0;
                const uint32_t lo = (uint32_t)m, hi = (uint32_t)(m >> 32);
                for (int cy = y0; cy <= y1; ++cy) {
                    if (lo) atomicOr(occ_s + 2 * cy, lo);
                    if (hi) atomicOr(occ_s + 2 * cy + 1, hi);
                }
            }
        } else {
            const int W = g.W;
            for (uint32_t t = lane; t < cnt; t += 32) {
                const int4 q = rq[t];
                if (q.x != 0) { hasx = 1; lox = min(lox, q.x); hix = max(hix, q.x); } else border = 1;
                if (q.z != W) { hasx = 1; lox = min(lox, q.z); hix = max(hix, q.z); } else border = 1;
                if (q.y != 0) { hasy = 1; loy = min(loy, q.y); hiy = max(hiy, q.y); } else border = 1;
                if (q.w != W) { hasy = 1; loy = min(loy, q.w); hiy = max(hiy, q.w); } else border = 1;
            }
            // rectangles by ascending area (ties by index): rank by counting
            for (uint32_t t = lane; t < cnt; t += 32) {
                if (nr > CHUNK) break;  // order_many
                const long long at = areas[t];  // before t: smaller areas, and equal ones of smaller index
                uint32_t rank = 0;
#pragma unroll 4
                for (uint32_t m = 0; m < nr; ++m) rank += areas[m] < at + (m < t ? 1 : 0) ? 1u : 0u;
                cs.rorder[r0 + rank] = (uint16_t)t;
            }
        }
    }
    if (nr > CHUNK) order_many<T, CHUNK>(r4, nr, areas, cs.rorder + r0);
    if (warp == 0) {
        hasx = __reduce_or_sync(0xffffffffu, hasx);
        hasy = __reduce_or_sync(0xffffffffu, hasy);
        border = __reduce_or_sync(0xffffffffu, border);
        lox = __reduce_min_sync(0xffffffffu, lox);
        hix = __reduce_max_sync(0xffffffffu, hix);
        loy = __reduce_min_sync(0xffffffffu, loy);
        hiy = __reduce_max_sync(0xffffffffu, hiy);
        if (lane == 0) {
            int4 *e = reinterpret_cast<int4 *>(cs.esig + (size_t)c * 8);
            e[0] = make_int4((int)nr, hasx, hasx ? lox : 0, hasx ? hix : 0);  // ES_N, ES_HASX, ES_LOX, ES_HIX
            e[1] = make_int4(hasy, hasy ? loy : 0, hasy ? hiy : 0, border);   // ES_HASY, ES_LOY, ES_HIY, ES_BORDER
            if (cs.spec_state) cs.spec_state[c] = 0;
        }
    }
    __syncthreads();
    // rows out (16 bytes a thread), row counts and the total
    uint32_t tot = 0;
    for (int j = tid; j < N; j += T) {
        uint32_t n = 0;
#pragma unroll
        for (int w = 0; w < W32; ++w) n += (uint32_t)__popc(rows[j * SR + w]);
        cs.prof[(size_t)c * 2 * N + j] = (uint16_t)n;
        tot += n;
    }
    tot = __reduce_add_sync(0xffffffffu, tot);
    if (lane == 0) red[warp] = tot;
    if constexpr (NW >= 2) {
        uint4 *dst = reinterpret_cast<uint4 *>(cs.bits + (size_t)c * N * NW);
        for (int t = tid; t < N * W32 / 4; t += T) {
            const uint32_t *w = rows + (t / (W32 / 4)) * SR + 4 * (t % (W32 / 4));
            dst[t] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        uint2 *dst = reinterpret_cast<uint2 *>(cs.bits + (size_t)c * N * NW);
        for (int t = tid; t < N; t += T) dst[t] = make_uint2(rows[t * SR], rows[t * SR + 1]);
    }
    for (int t = tid; t < 64; t += T)
        cs.occ[(size_t)c * 64 + t] = (uint64_t)occ_s[2 * t] | ((uint64_t)occ_s[2 * t + 1] << 32);
    __syncthreads();
    tot = 0;
#pragma unroll
    for (int k = 0; k < T / 32; ++k) tot += red[k];
    if (tid == 0) cs.pop[c] = tot;
    uint16_t *cols = cs.prof + (size_t)c * 2 * N + N;
    if (tot == area_sum) {
        // no shared pixel: column counts by a prefix sum (lane l: N / 32 columns)
        if (warp == 0) {
            constexpr int K = N / 32;
            int v[K], s = 0;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                s += diff[K * lane + k];
                v[k] = s;
            }
            int x = s;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            x -= s;
            __syncwarp();  // all differences are read: the counts take their place
#pragma unroll
            for (int k = 0; k < K; ++k) reinterpret_cast<uint16_t *>(diff)[K * lane + k] = (uint16_t)(x + v[k]);
            __syncwarp();
            for (int t = lane; t < N; t += 32) cols[t] = reinterpret_cast<const uint16_t *>(diff)[t];
        }
    } else {
        // counted from the rows: each column's ones, each block's
        for (int i = tid; i < N; i += T) {
            uint32_t n = 0;
            for (int j = 0; j < N; ++j) n += (rows[j * SR + (i >> 5)] >> (i & 31)) & 1u;
            cols[i] = (uint16_t)n;
        }
        for (int t = tid; t < NB2; t += T) {
            const int by = t / NB, bx = t % NB;
            uint32_t n = 0;
            for (int j = 0; j < 16; ++j)
                n += (uint32_t)__popc((rows[(16 * by + j) * SR + (bx >> 1)] >> (16 * (bx & 1))) & 0xffffu);
            cnt_s[t] = n;
        }
        __syncthreads();
    }
    // 16x16 block counts, then neighbourhood sums, each stored in the order of
    // blk_pos: blocks spread over the whole clip come first, so the gates'
    // chunked density bound sees every part of the clip in its first chunk;
    // the sums by rows, then by columns (nbh: over the rows [by - rb, by + rb])
    uint32_t *nbh = rows;  // the rows are written
    static_assert(N * SR >= NB2, "room for the row sums");
    __syncthreads();
    const int rb = g.rb;
    for (int t = tid; t < NB2; t += T) {
        const int by = t / NB;
        uint32_t s = cnt_s[t];
        if (rb == 1) {
            s += (by > 0 ? cnt_s[t - NB] : 0u) + (by < NB - 1 ? cnt_s[t + NB] : 0u);
        } else {
            for (int d = 1; d <= rb; ++d)
                s += (by >= d ? cnt_s[t - d * NB] : 0u) + (by + d < NB ? cnt_s[t + d * NB] : 0u);
        }
        nbh[t] = s;
    }
    __syncthreads();
    uint16_t *blk = cs.blk + (size_t)c * 2 * NB2;
    constexpr int Q = NB / 4, QQ = Q * Q;
    for (int t = tid; t < NB2; t += T) {  // t: position of a block in the stored order
        const int grp = t / QQ, by = ((t % QQ) / Q) * 4 + (grp >> 2), bx = (t % Q) * 4 + (grp & 3);
        const uint32_t *at = nbh + by * NB + bx;
        uint32_t s = at[0];
        if (rb == 1) {
            s += (bx > 0 ? at[-1] : 0u) + (bx < NB - 1 ? at[1] : 0u);
        } else {
            for (int d = 1; d <= rb; ++d) s += (bx >= d ? at[-d] : 0u) + (bx + d < NB ? at[d] : 0u);
        }
        blk[t] = (uint16_t)cnt_s[by * NB + bx];
        blk[NB2 + t] = (uint16_t)min(s, 65535u);
    }
}

}  // namespace

cudaError_t launch_raster(const pcl_params &prm, const pcl_clipset &cs, cudaStream_t st) {
    const Geo g = make_geo(prm);
    if (cs.n_clips == 0) return cudaSuccess;
    const unsigned grid = cs.n_clips;
    switch (g.nw) {
        case 1: raster_kernel<1><<<grid, RasterCta<1>::threads, 0, st>>>(prm, cs); break;
        case 2: raster_kernel<2><<<grid, RasterCta<2>::threads, 0, st>>>(prm, cs); break;
        case 4: raster_kernel<4><<<grid, RasterCta<4>::threads, 0, st>>>(prm, cs); break;
        case 8: raster_kernel<8><<<grid, RasterCta<8>::threads, 0, st>>>(prm, cs); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace pcl
