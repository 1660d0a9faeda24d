// b = 1 gather with X in shared memory (static GATHER plans, where the estimate in
// gather_xs_takes is clearly below the row items' kernels).
//
// The gather kernel (k_cudacore.cu) fetches a row of X from L2 for every
// non-zero: at n = 32 that is 64 bytes per 4-byte non-zero, and L2's latency
// and random-access rate bound it.  Here a cluster of CS CTAs covers k, each
// CTA copies its slice of X (its rows x NC columns) into shared memory once and
// walks a range of W's rows; a warp takes one row of the slice at a time,
// streams its 16-bit column indices and values (32 per load, up to 128 in
// flight, the next row's requested ahead), hands one non-zero to each group of
// LN lanes by a shuffle, and every lane multiplies its 16 bytes of that X row
// (V columns) in FP32.  The groups' sums meet in fixed exchanges, the row's sum
// over the slice stays in shared memory, and after a cluster barrier each CTA
// adds its share of the rows over the slices in order (distributed shared
// memory) and writes Y: no partial sums in memory and one launch.
//
// Bound: issue (a shuffle, a 16-byte shared load and V mixed-precision FMAs per
// non-zero and lane, fma16.cuh) and shared-memory wavefronts (two random 64-byte rows per
// quarter warp at n = 32: 1.5 each on average).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "fma16.cuh"
#include "pdl.cuh"
#include "spmm_internal.h"

namespace spmm {
namespace {

constexpr int kGxWarps = 16;
constexpr int kGxSmem = 220 * 1024;
constexpr int kGxU = 4;                  // loads of 32 non-zeros in flight

// A non-zero as the lanes hand it on: column and weight, one word (and one
// shuffle) for 16-bit values.  V: columns per lane, 16 bytes of X.
template <typename T> struct Gx {
    static constexpr int V = 8;
    using Nz = uint32_t;
    static __device__ __forceinline__ Nz nz(uint16_t c, T v) {
        return c | (uint32_t)*reinterpret_cast<const uint16_t *>(&v) << 16;
    }
    static __device__ __forceinline__ void from_lane(Nz z, int lane, uint32_t &c, T &w) {
        z = __shfl_sync(0xffffffffu, z, lane);
        c = z & 0xFFFFu;
        const uint16_t h = (uint16_t)(z >> 16);
        w = *reinterpret_cast<const T *>(&h);
    }
};
template <> struct Gx<float> {
    static constexpr int V = 4;
    struct Nz {
        uint32_t c;
        float w;
    };
    static __device__ __forceinline__ Nz nz(uint16_t c, float v) { return {c, v}; }
    static __device__ __forceinline__ void from_lane(Nz z, int lane, uint32_t &c, float &w) {
        c = __shfl_sync(0xffffffffu, z.c, lane);
        w = __shfl_sync(0xffffffffu, z.w, lane);
    }
};
__device__ __forceinline__ float gx_out(float v, float) { return v; }
__device__ __forceinline__ __half gx_out(float v, __half) { return __float2half_rn(v); }
__device__ __forceinline__ __nv_bfloat16 gx_out(float v, __nv_bfloat16) {
    return __float2bfloat16_rn(v);
}
template <typename T, int V> __device__ __forceinline__ void gx_fma(float *acc, uint4 x, T w) {
    const T *xv = reinterpret_cast<const T *>(&x);
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = fma16(w, xv[v], acc[v]);
}

struct GxArgs {
    const int32_t *ptr;          // first non-zero of (row, part of k); kGxParts per row
    const uint16_t *col;
    const void *vals, *X;
    void *Y;
    int64_t ldx, ldy, n, m, k;
    int32_t pw;                  // columns of W per part
    int32_t rr, rp;              // rows per unit, per pass
    int32_t nchunk, poff, xvec;  // column chunks; partials' offset; X rows 16-byte aligned
};

__device__ __forceinline__ float4 gx_remote(uint32_t addr, int rank) {
    uint32_t a;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}
__device__ __forceinline__ void gx_cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T, int LN, int CS>
__global__ void __launch_bounds__(kGxWarps * 32, 1) gather_xs_kernel(const GxArgs A) {
    pdl_enter();
    constexpr int V = Gx<T>::V, NC = LN * V, G = 32 / LN;
    constexpr int SB = NC * (int)sizeof(T);              // bytes of an X row in shared memory
    extern __shared__ __align__(128) uint8_t gx_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const int unit = (int)(blockIdx.x / CS), range = unit / A.nchunk, chunk = unit - range * A.nchunk;
    const int64_t row0 = (int64_t)range * A.rr;
    const int rows = (int)min((int64_t)A.rr, A.m - row0);
    const int c0 = chunk * NC;
    constexpr int kPer = kGxParts / CS;
    const int part0 = (int)rank * kPer;
    const int64_t k0 = min((int64_t)part0 * A.pw, A.k), k1 = min(k0 + (int64_t)kPer * A.pw, A.k);
    const int nv = (int)min((int64_t)NC, A.n - c0);      // columns of X here
    const T *X = reinterpret_cast<const T *>(A.X) + k0 * A.ldx + c0;
    const uint32_t sx = (uint32_t)__cvta_generic_to_shared(gx_smem);
    // ---- the slice of X, columns past n zero
    if (A.xvec) {
        for (int i = tid; i < (int)(k1 - k0) * LN; i += kGxWarps * 32) {
            const int r = i / LN, c = i % LN, left = nv - c * V;
            const int bytes = left >= V ? 16 : left > 0 ? left * (int)sizeof(T) : 0;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sx + i * 16),
                         "l"(bytes ? X + (int64_t)r * A.ldx + c * V : X), "r"(bytes)
                         : "memory");
        }
    } else {
        T *xs = reinterpret_cast<T *>(gx_smem);
        for (int i = tid; i < (int)(k1 - k0) * NC; i += kGxWarps * 32) {
            const int r = i / NC, c = i % NC;
            xs[i] = c < nv ? X[(int64_t)r * A.ldx + c] : gx_out(0.f, T());
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    float *part = reinterpret_cast<float *>(gx_smem + A.poff);
    const int sg = lane / LN, lc = lane % LN;
    const T *vals = reinterpret_cast<const T *>(A.vals);
    const uint8_t *xl = gx_smem + lc * 16 - k0 * SB;     // + column x SB: this lane's piece
    for (int base = 0; base < rows; base += A.rp) {
        const int prows = min(A.rp, rows - base);
        auto range_of = [&](int r, int32_t &b, int32_t &e) {
            b = e = 0;
            if (r < prows) {
                const int32_t *p = A.ptr + (row0 + base + r) * kGxParts + part0;
                b = __ldg(p);
                e = __ldg(p + kPer);
            }
        };
        // 32 kGxU non-zeros from i: index and value of non-zero i + 32 u + lane
        uint16_t cn[kGxU];
        T vn[kGxU];
        auto load = [&](int32_t i, int32_t e) {
#pragma unroll
            for (int u = 0; u < kGxU; ++u) {
                const int32_t j = i + 32 * u + lane;
                cn[u] = j < e ? __ldg(A.col + j) : (uint16_t)0;
                vn[u] = j < e ? vals[j] : gx_out(0.f, T());
            }
        };
        int r = warp;
        int32_t b, e, nb, ne;
        range_of(r, b, e);
        range_of(r + kGxWarps, nb, ne);
        load(b, e);
        if (base == 0) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();                              // the X slice is here
        }
        for (; r < prows; r += kGxWarps) {
            float acc[V];
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] = 0.f;
            int32_t n2b, n2e;
            range_of(r + 2 * kGxWarps, n2b, n2e);
            for (int32_t i = b; i < e; i += 32 * kGxU) {
                typename Gx<T>::Nz z[kGxU];
#pragma unroll
                for (int u = 0; u < kGxU; ++u) z[u] = Gx<T>::nz(cn[u], vn[u]);
                const int cnt = e - i;
                // the next 128 of this row, or the next row's first, on the way
                if (cnt > 32 * kGxU) load(i + 32 * kGxU, e);
                else load(nb, ne);
#pragma unroll
                for (int u = 0; u < kGxU; ++u) {
                    // group sg takes non-zeros sg, sg + G, ... of these 32; all
                    // 32 there: the loads of a batch go out together
                    if (32 * (u + 1) <= cnt) {
                        constexpr int NB = LN < 4 ? LN : 4;
#pragma unroll
                        for (int t0 = 0; t0 < LN; t0 += NB) {
                            uint32_t c[NB];
                            T w[NB];
                            uint4 x[NB];
#pragma unroll
                            for (int t = 0; t < NB; ++t)
                                Gx<T>::from_lane(z[u], (t0 + t) * G + sg, c[t], w[t]);
#pragma unroll
                            for (int t = 0; t < NB; ++t)
                                x[t] = *reinterpret_cast<const uint4 *>(xl + c[t] * SB);
#pragma unroll
                            for (int t = 0; t < NB; ++t) gx_fma<T, V>(acc, x[t], w[t]);
                        }
                    } else if (32 * u < cnt) {
#pragma unroll
                        for (int t = 0; t < LN; ++t) {
                            const int j = t * G + sg;
                            uint32_t c;
                            T w;
                            Gx<T>::from_lane(z[u], j, c, w);
                            if (32 * u + j < cnt)
                                gx_fma<T, V>(acc, *reinterpret_cast<const uint4 *>(xl + c * SB), w);
                        }
                    }
                }
            }
            if (b >= e) load(nb, ne);                     // (an empty row loaded nothing)
            b = nb, e = ne, nb = n2b, ne = n2e;
            // the groups' sums: each exchange halves the values a lane keeps, so a
            // row takes 7 shuffles at n = 32 where a butterfly takes 24
            int keep = V, at = 0, dup = 0;
#pragma unroll
            for (int off = LN; off < 32; off <<= 1) {
                if (keep > 1) {
                    keep /= 2;
                    const bool up = lane & off;
#pragma unroll
                    for (int v = 0; v < V / 2; ++v) {
                        if (v < keep) {
                            const float mine = up ? acc[keep + v] : acc[v];
                            const float other = up ? acc[v] : acc[keep + v];
                            acc[v] = mine + __shfl_xor_sync(0xffffffffu, other, off);
                        }
                    }
                    at += up ? keep : 0;
                } else {
                    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
                    dup |= lane & off;
                }
            }
            if (!dup) {
                float *d = part + r * NC + lc * V + at;
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (v < keep) d[v] = acc[v];
            }
        }
        gx_cluster_sync();
        // this CTA's rows of the pass, over the slices in order
        constexpr int Q = NC / 4;
        const uint32_t sp = sx + A.poff;
        for (int i = tid; i < (prows + CS - 1) / CS * Q; i += kGxWarps * 32) {
            const int rr = (i / Q) * CS + (int)rank, c = (i % Q) * 4;
            if (rr >= prows || c >= nv) continue;
            float4 v[CS], s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < CS; ++q) v[q] = gx_remote(sp + (rr * NC + c) * 4, q);
#pragma unroll
            for (int q = 0; q < CS; ++q) s.x += v[q].x, s.y += v[q].y, s.z += v[q].z, s.w += v[q].w;
            T *y = reinterpret_cast<T *>(A.Y) + (row0 + base + rr) * A.ldy + c0 + c;
            const float o[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c + q < nv) y[q] = gx_out(o[q], T());
        }
        gx_cluster_sync();       // peers may still read this CTA's partials
    }
}

// Clusters of CS CTAs that run at once (one CTA per SM).
template <int CS> int gx_clusters() {
    static std::atomic<int> known{0};
    int c = known.load(std::memory_order_relaxed);
    if (c) return c;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS);
    cfg.blockDim = dim3(kGxWarps * 32);
    cfg.dynamicSmemBytes = kGxSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto kernel = gather_xs_kernel<__half, 1, CS>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGxSmem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&c, kernel, &cfg) != cudaSuccess || c < 1)
        c = 128 / CS;
    known.store(c, std::memory_order_relaxed);
    return c;
}

template <typename T, int LN, int CS>
cudaError_t gx_launch(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, void *Y,
                      int64_t ldy, cudaStream_t s) {
    constexpr int NC = LN * Gx<T>::V;
    GxArgs A;
    A.ptr = p->d_gx_ptr;
    A.col = p->d_col16;
    A.vals = p->d_packed;
    A.X = X;
    A.Y = Y;
    A.ldx = ldx;
    A.ldy = ldy;
    A.n = n;
    A.m = p->m;
    A.k = p->k;
    A.pw = (int32_t)((p->k + kGxParts - 1) / kGxParts);
    A.nchunk = (int32_t)((n + NC - 1) / NC);
    A.xvec = (uintptr_t)X % 16 == 0 && ldx * (int64_t)sizeof(T) % 16 == 0 ? 1 : 0;
    A.poff = kGxParts / CS * A.pw * NC * (int)sizeof(T);
    const int64_t ranges = std::max<int64_t>(1, gx_clusters<CS>() / A.nchunk);
    A.rr = (int32_t)((p->m + ranges - 1) / ranges);
    const int room = (kGxSmem - A.poff) / (NC * 4);
    const int np = (A.rr + room - 1) / room;
    A.rp = (A.rr + np - 1) / np;
    const int64_t units = (p->m + A.rr - 1) / A.rr * A.nchunk;
    if (units * CS > INT32_MAX) return cudaErrorInvalidConfiguration;
    static std::atomic<uint64_t> attrs{0};
    cudaError_t e = set_smem_attrs_once(attrs, gather_xs_kernel<T, LN, CS>, kGxSmem, true);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(units * CS));
    cfg.blockDim = dim3(kGxWarps * 32);
    cfg.dynamicSmemBytes = (size_t)A.poff + (size_t)A.rp * NC * 4;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CS;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, gather_xs_kernel<T, LN, CS>, A);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// Lanes per X row (a power of two whose columns cover n, at most 8) and CTAs
// per cluster: the fewest that hold X, at most four; then fewer columns.
template <typename T> bool gx_shape(const spmm_plan *p, int64_t n, int *ln, int *cs) {
    constexpr int V = Gx<T>::V;
    int l = 1;
    while (l < 8 && l * V < n) l *= 2;
    const int64_t pw = (p->k + kGxParts - 1) / kGxParts;
    for (; l >= 1; l /= 2)
        for (int c = 1; c <= 4; c *= 2)
            if (kGxParts / c * pw * l * 16 + 16 * l * V * 4 <= kGxSmem) {
                *ln = l;
                *cs = c;
                return true;
            }
    return false;
}

template <typename T>
cudaError_t gx_dispatch(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, void *Y,
                        int64_t ldy, cudaStream_t s) {
    int ln = 0, cs = 0;
    if (!gx_shape<T>(p, n, &ln, &cs)) return cudaErrorInvalidConfiguration;
    switch (ln * 8 + cs) {
        case 8 + 1: return gx_launch<T, 1, 1>(p, X, n, ldx, Y, ldy, s);
        case 8 + 2: return gx_launch<T, 1, 2>(p, X, n, ldx, Y, ldy, s);
        case 8 + 4: return gx_launch<T, 1, 4>(p, X, n, ldx, Y, ldy, s);
        case 16 + 1: return gx_launch<T, 2, 1>(p, X, n, ldx, Y, ldy, s);
        case 16 + 2: return gx_launch<T, 2, 2>(p, X, n, ldx, Y, ldy, s);
        case 16 + 4: return gx_launch<T, 2, 4>(p, X, n, ldx, Y, ldy, s);
        case 32 + 1: return gx_launch<T, 4, 1>(p, X, n, ldx, Y, ldy, s);
        case 32 + 2: return gx_launch<T, 4, 2>(p, X, n, ldx, Y, ldy, s);
        case 32 + 4: return gx_launch<T, 4, 4>(p, X, n, ldx, Y, ldy, s);
        case 64 + 1: return gx_launch<T, 8, 1>(p, X, n, ldx, Y, ldy, s);
        case 64 + 2: return gx_launch<T, 8, 2>(p, X, n, ldx, Y, ldy, s);
        default: return gx_launch<T, 8, 4>(p, X, n, ldx, Y, ldy, s);
    }
}

}  // namespace

// Whether this kernel takes a call, or the row items' kernels (k_cudacore.cu)
// keep it.  Either can be several times as fast: this one copies all of X's
// slice into every CTA and walks equal ranges of rows, so few non-zeros per row,
// or a pattern that loads one range, one slice or one row, leave it waiting;
// the item kernels fetch a row of X per non-zero, from items cut to length.  So
// both times are estimated, and this kernel has to promise 15 % less.  The
// terms were fitted to products timed with both kernels on a GB300 (m 100 to
// 16384, k 100 to 53000, n 1 to 300, d 1/4 to 1/4096; uniform, banded, diagonal
// and skewed patterns).  On 1411 of them the estimates' rms errors are 10 to 21
// %, the pick takes 1.04 times the faster kernel's time on average, and it is
// more than 3 % slower than the items once (0.92 of their speed).  us, items -> this:
// d = 1/16, FP16, 8192 x 8192: n = 12 29.5 -> 17.0, n = 32 43.2 -> 25.0, n = 100 181
// -> 87; 4096 x 4096, d = 1/8, n = 64: 66.2 -> 20.0, FP32 58.6 -> 32.4.  Kept by
// the items: 8192 x 8192, d = 1/1024, n = 100: 7.4 (48.0 here); 4096 x 4096, d =
// 1/256, FP32, n = 64: 5.8 (15.4); 2048 x 2048, d = 1/64, n = 20: 3.9 (8.0); 4096 x
// 4096, d = 1/16 near the diagonal, FP32, n = 64: 27.9 (53.4).
static double gx_us(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, int ln, int cs) {
    const bool f32 = p->xdt == SPMM_F32;
    const int es = f32 ? 4 : 2, V = 16 / es, c = cs >> 1;   // c = log2 cs
    // (host-only plans make no CUDA calls: a GB300's 152 SMs)
    const int64_t cl = p->host_only ? (cs == 4 ? 36 : 152 / cs)
                       : cs == 1    ? gx_clusters<1>()
                       : cs == 2    ? gx_clusters<2>()
                                    : gx_clusters<4>();
    const int64_t nch = (n + ln * V - 1) / (ln * V), ranges = std::max<int64_t>(1, cl / nch);
    const int64_t rr = (p->m + ranges - 1) / ranges;
    const double waves = (double)(((p->m + rr - 1) / rr * nch + cl - 1) / cl);
    int j = 0;
    while (j < 7 && (2 << j) <= ranges) ++j;
    const double heavy = std::max((double)p->gx.heavy[c][j] * (double)(1 << j) / (double)ranges,
                                  (1 << j) < ranges ? (double)p->gx.heavy[c][std::min(j + 1, 7)] : 0);
    // X: 16-byte pieces (rows of an odd number of them are slow to copy), or
    // values one by one
    const double pieces = (double)p->k / cs * ln;
    const int64_t row = ldx * es;
    const double copy = (uintptr_t)X % 16 || row % 16 ? 1.45e-4 * V
                        : row % 32 && ln > 1          ? 6.7e-4
                                                      : f32 ? 1.75e-4 : 1.9e-4;
    const double rows = (double)rr, slice = (double)p->gx.row_slice[c];
    return (f32 ? 3.13 : 2.95) +
           waves * (pieces * copy + rows / 16 * (f32 ? 0.555 : 0.57) +
                    rows * ln * (f32 ? 4.5e-4 : 1.8e-3) +
                    heavy * (f32 ? 6.6e-5 * ln + 1.1e-4 : 3.95e-5 * ln + 1.5e-4) +
                    slice * (f32 ? 2.5e-4 * ln + 1e-3 : 5e-4 * ln + 1.2e-3));
}

static double items_us(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, const void *Y,
                       int64_t ldy) {
    const bool f32 = p->xdt == SPMM_F32;
    const double nnz = (double)p->nnzb, reds = (double)p->n_red;
    const double item = (double)std::min<int64_t>(p->gx.longest_row, p->C);
    const int64_t vecs = n / gather_vector(p, X, n, ldx, Y, ldy);
    if (vecs == 1)   // gather1g_kernel (16-bit values)
        return 3.5 + nnz * (1.05e-6 + 2.2e-8 * (double)n) + 0.0037 * item + 4.4e-4 * (double)p->m +
               (reds > 0 ? 2.2 + 0.036 * reds : 0);
    int64_t ln = 1;
    while (ln < 32 && ln < vecs) ln *= 2;
    const double nch = (double)((vecs + ln - 1) / ln);
    return (f32 ? 2.18 : 2.3) + 2.3e-4 * (double)p->n_items * nch +
           nnz * ((f32 ? 4.7e-7 : 3.0e-7) * (double)ln * nch +
                  (double)n * (f32 ? 4 * 3.5e-8 : 2 * 1.75e-7)) +
           item * (0.0015 * (double)ln + (f32 ? 0.0046 : 0.0042)) +
           (reds > 0 ? 2.0 + 0.015 * reds * (double)((n + 127) / 128) : 0);
}

bool gather_xs_takes(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, const void *Y,
                     int64_t ldy) {
    if (!p->gx.on || n < 1) return false;
    int ln, cs;
    if (p->xdt == SPMM_F32) {
        // more than one vector per row, and a slice that holds as many columns
        // as one warp covers
        int cover = 1;
        while (cover < 8 && cover * 4 < n) cover *= 2;
        if (n <= 4 || !gx_shape<float>(p, n, &ln, &cs) || ln != cover) return false;
    } else {
        if (!gx_shape<__half>(p, n, &ln, &cs)) return false;
    }
    // one vector of X per row that fits the ring kernel's memory: that kernel
    // (8192 x 8192, n = 1: 8.3 against 13.5 us)
    if (gather_vector(p, X, n, ldx, Y, ldy) == n && gather_ring_fits(p, n)) return false;
    return gx_us(p, X, n, ldx, ln, cs) < 0.85 * items_us(p, X, n, ldx, Y, ldy);
}

cudaError_t launch_gather_xs(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, void *Y,
                             int64_t ldy, cudaStream_t s) {
    switch (p->xdt) {
        case SPMM_F32: return gx_dispatch<float>(p, X, n, ldx, Y, ldy, s);
        case SPMM_F16: return gx_dispatch<__half>(p, X, n, ldx, Y, ldy, s);
        case SPMM_BF16: return gx_dispatch<__nv_bfloat16>(p, X, n, ldx, Y, ldy, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace spmm
