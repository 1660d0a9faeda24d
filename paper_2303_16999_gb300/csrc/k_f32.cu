// FP32 product of b x b blocks, b in {4, 8, 16} (Section 3's product on the
// CUDA cores; what AUTO plans with FP32 W and X run).
//
// A CTA of KS warps owns one block row and one chunk of columns; warp w takes
// blocks w, w + KS, ... of the row and keeps the chunk's partial outputs in
// registers: lanes are (row part, column group), a lane holds b / RS rows x
// kF32Cols columns.  Every X value a warp brings in serves all b rows of the
// block row, where one thread per output reads it once per row: that and the
// serial chain of two loads per FMA held the plain kernel at 4.7 TFLOP/s.  X
// comes straight into registers, F32Cfg::D stages of F32Cfg::NL rows ahead;
// W blocks (stored column by column, so a lane reads the rows of one column of
// W in 16-byte pieces, the same address in every lane of a row part) pass
// through a per-warp cp.async ring.  The warps meet once, at the end, where
// their partials are added in warp order.
//
// FMAs are packed in pairs of rows (two of W's rows arrive in adjacent
// registers; x is duplicated), which leaves issue slots for the loads.
// Measured against the plain kernel: 2048 x 4096, b = 8, d = 1/8, n = 500: 220
// -> 32 us (33 TFLOP/s); 4096 x 4096, n = 1024, d = 1/16: b = 16 323 -> 52 us,
// b = 4 605 -> 77 us (X at 13.9 TB/s).  One warp per block row and chunk, with
// the plain kernel's order of sums, took 53 us on the first: too few warps to
// cover the loads' latency.
// Bound: the FMAs and X through L2 and L1 (b * chunk * 4 bytes per block and
// chunk; at b = 4 that traffic alone).
#include <cuda_runtime.h>

#include "pdl.cuh"
#include "spmm_internal.h"

namespace spmm {
namespace {

constexpr int kF32Cols = 4;      // columns per lane

__device__ __forceinline__ void f32_cp(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
// (a.x, a.y) += (w.x x, w.y x), each rounded as a scalar fmaf would be.
__device__ __forceinline__ void f32_fma2(float2 &a, float2 w, float x) {
    unsigned long long av, wv, xv, d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(av) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(wv) : "f"(w.x), "f"(w.y));
    asm("mov.b64 %0, {%1, %1};" : "=l"(xv) : "f"(x));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(wv), "l"(xv), "l"(av));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(d));
}

// NL: X rows per register stage (a block; a quarter or half of one at b =
// 16); D: register stages, D - 1 of them in flight while one is multiplied;
// S: W blocks in a warp's ring.
template <int B, int RS> struct F32Cfg {
    static constexpr int NL = B == 16 && RS == 1 ? 4 : B == 4 ? 4 : 8;
    static constexpr int D = B == 4 ? 4 : B == 16 && RS == 1 ? 3 : 2;
    static constexpr int S = 4;
    // CTAs per SM the registers are held to: 16 warps at most 128 each (at
    // 132, one CTA fewer per SM, the b = 8 product below took 37.4 us)
    static constexpr int kCtas = B == 16 && RS == 1 ? 3 : RS > 2 ? 2 : 4;
};

// B: block size.  RS: lanes that share a column group, each with B / RS rows
// of the block row (1 for n > 64; for fewer columns the lanes split the
// rows, so few stay idle).  KS: warps per CTA.  VEC: X rows are 16-byte
// aligned, a lane's columns are consecutive; else they lie 32 / RS apart, so
// loads stay coalesced.
template <int B, int RS, int KS, bool VEC>
__global__ void __launch_bounds__(KS * 32, F32Cfg<B, RS>::kCtas)
    f32_block_kernel(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col_idx,
                     const float *__restrict__ vals, const float *__restrict__ X, int64_t ldx,
                     float *__restrict__ Y, int64_t ldy, int64_t n, int nchunk, int yvec) {
    pdl_enter();
    using G = F32Cfg<B, RS>;
    constexpr int L = 32 / RS;                  // column groups
    constexpr int RL = B / RS;                  // rows per lane
    constexpr int CH = L * kF32Cols;            // columns per CTA
    constexpr int NL = G::NL, D = G::D, S = G::S;
    constexpr int H = B / NL;                   // register stages per block
    constexpr int kWPieces = B * B / 4;         // 16-byte pieces of a W block
    constexpr int kRing = S * B * B, kPart = RL * kF32Cols * 32;
    // the warps' rings, then (after the last block) their partials
    __shared__ __align__(16) float smem[KS * (kRing > kPart ? kRing : kPart)];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *ring = smem + warp * kRing;
    const int64_t r = blockIdx.x / (unsigned)nchunk;
    const int64_t c0 = (int64_t)(blockIdx.x % (unsigned)nchunk) * CH;
    const int lc = lane % L, lr = lane / L;
    // column v of this lane: cx + v * CS, inside X while v < cnt
    constexpr int CS = VEC ? 1 : L;
    const int64_t cx = c0 + (VEC ? lc * kF32Cols : lc);
    const int cnt = n <= cx ? 0 : (int)min((int64_t)kF32Cols, (n - cx + CS - 1) / CS);
    const float *xlane = X + (cnt ? cx : 0);
    const int32_t beg = row_ptr[r], all = row_ptr[r + 1] - beg;
    // this warp's blocks: CSR slots beg + warp + KS * q, q < nblk
    const int nblk = all > warp ? (all - warp + KS - 1) / KS : 0;
    const int nst = nblk * H;
    vals += ((int64_t)beg + warp) * (B * B);
    col_idx += beg + warp;
    // block columns of 32 blocks, one per lane, the next 32 requested ahead
    int32_t cols = lane < nblk ? col_idx[lane * KS] : 0;
    int32_t cols_next = 32 + lane < nblk ? col_idx[(32 + lane) * KS] : 0;
    float4 xr[D][NL];
    // rows of register stage t (part t % H of block t / H), in order of t
    auto load = [&](int t, float4 *x) {
        if (t >= nst) return;
        const int q = t / H, h = t % H;
        if (h == 0 && q > 0 && (q & 31) == 0) {
            cols = cols_next;
            cols_next = q + 32 + lane < nblk ? col_idx[(q + 32 + lane) * KS] : 0;
        }
        const int64_t c = __shfl_sync(0xffffffffu, cols, q & 31);
        const float *xs = xlane + (c * B + h * NL) * ldx;
        if (VEC && cnt == kF32Cols) {
#pragma unroll
            for (int l = 0; l < NL; ++l)
                x[l] = __ldg(reinterpret_cast<const float4 *>(xs + l * ldx));
        } else {
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                x[l].x = cnt > 0 ? __ldg(xs + l * ldx) : 0.f;
                x[l].y = cnt > 1 ? __ldg(xs + l * ldx + CS) : 0.f;
                x[l].z = cnt > 2 ? __ldg(xs + l * ldx + 2 * CS) : 0.f;
                x[l].w = cnt > 3 ? __ldg(xs + l * ldx + 3 * CS) : 0.f;
            }
        }
    };
    auto load_w = [&](int q) {
        if (q < nblk) {
            float *st = ring + (q % S) * (B * B);
            const float *src = vals + (int64_t)q * (KS * B * B);
#pragma unroll
            for (int w = 0; w < (kWPieces + 31) / 32; ++w)
                if (kWPieces % 32 == 0 || w * 32 + lane < kWPieces)
                    f32_cp(st + (w * 32 + lane) * 4, src + (w * 32 + lane) * 4);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int q = 0; q < S - 1; ++q) load_w(q);
#pragma unroll
    for (int d = 0; d < D; ++d) load(d, xr[d]);
    constexpr int RP = (RL + 1) / 2;            // row pairs (RL = 1: one row, .y unused)
    float2 acc[RP][kF32Cols];
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int v = 0; v < kF32Cols; ++v) acc[i][v] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int t0 = 0; t0 < nst; t0 += D) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int t = t0 + d;
            if (t >= nst) break;
            const int q = t / H, h = t % H;
            if (h == 0) {
                asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
                __syncwarp();    // W block q has landed; every lane is past block q - 1
                load_w(q + S - 1);
            }
            const float *wr = ring + (q % S) * (B * B) + h * NL * B + lr * RL;
#pragma unroll
            for (int l = 0; l < NL; ++l) {
                const float xv[4] = {xr[d][l].x, xr[d][l].y, xr[d][l].z, xr[d][l].w};
                if constexpr (RL == 1) {
                    const float w = wr[l * B];
#pragma unroll
                    for (int v = 0; v < kF32Cols; ++v) acc[0][v].x = fmaf(w, xv[v], acc[0][v].x);
                } else {
                    float2 w[RP];
                    if constexpr (RL == 2) {
                        w[0] = *reinterpret_cast<const float2 *>(wr + l * B);
                    } else {
#pragma unroll
                        for (int i = 0; i < RL; i += 4) {
                            const float4 u = *reinterpret_cast<const float4 *>(wr + l * B + i);
                            w[i / 2] = make_float2(u.x, u.y);
                            w[i / 2 + 1] = make_float2(u.z, u.w);
                        }
                    }
#pragma unroll
                    for (int v = 0; v < kF32Cols; ++v)
#pragma unroll
                        for (int i = 0; i < RP; ++i) f32_fma2(acc[i][v], w[i], xv[v]);
                }
            }
            load(t + D, xr[d]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();             // every warp is past its ring
    float *part = smem + warp * kPart + lane;
#pragma unroll
    for (int i = 0; i < RL; ++i)
#pragma unroll
        for (int v = 0; v < kF32Cols; ++v)
            part[(i * kF32Cols + v) * 32] = i & 1 ? acc[i / 2][v].y : acc[i / 2][v].x;
    __syncthreads();
    if (cnt == 0) return;
    for (int i = warp; i < RL; i += KS) {
        float o[kF32Cols];
#pragma unroll
        for (int v = 0; v < kF32Cols; ++v) {
            const float *src = smem + lane + (i * kF32Cols + v) * 32;
            o[v] = src[0];
#pragma unroll
            for (int w = 1; w < KS; ++w) o[v] += src[w * kPart];
        }
        float *y = Y + (r * B + lr * RL + i) * ldy + cx;
        if (VEC && yvec && cnt == kF32Cols) {
            *reinterpret_cast<float4 *>(y) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int v = 0; v < kF32Cols; ++v)
                if (v < cnt) y[v * CS] = o[v];
        }
    }
}

template <int B, int RS, int KS>
cudaError_t f32_launch(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, void *Y,
                       int64_t ldy, cudaStream_t s) {
    constexpr int CH = 32 / RS * kF32Cols;
    const int64_t nchunk = (n + CH - 1) / CH, units = p->m / B * nchunk;
    if (units > INT32_MAX) return cudaErrorInvalidConfiguration;
    // b = 8, n > 64 takes spaced columns always: 32.1 us against 37.3 with
    // 16-byte loads (2048 x 4096, d = 1/8, n = 500), and 0.80 to 1.06 of their time over
    // 26 other products (256 to 4096, d = 1/32 and 1/4, n 128 to 500); b = 4 and 16
    // lose by them (77 -> 85 and 52 -> 60 us at 4096 x 4096, d = 1/16, n = 1024)
    constexpr bool kVec = !(B == 8 && RS == 1);
    const bool xvec = kVec && (uintptr_t)X % 16 == 0 && ldx % 4 == 0;
    const int yvec = (uintptr_t)Y % 16 == 0 && ldy % 4 == 0 ? 1 : 0;
    return pdl_launch(
        xvec ? f32_block_kernel<B, RS, KS, kVec> : f32_block_kernel<B, RS, KS, false>,
        dim3((unsigned)units), dim3(KS * 32), 0, s, (const int32_t *)p->d_row_ptr,
        (const int32_t *)p->d_col_idx, (const float *)p->d_packed, (const float *)X, ldx,
        (float *)Y, ldy, n, (int)nchunk, yvec);
}

template <int B>
cudaError_t f32_dispatch(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, void *Y,
                         int64_t ldy, cudaStream_t s) {
    // the narrowest warp whose columns cover n, down to four column groups
    if (n > 64) return f32_launch<B, 1, 4>(p, X, n, ldx, Y, ldy, s);
    if (n > 32) return f32_launch<B, 2, 4>(p, X, n, ldx, Y, ldy, s);
    if (n > 16 || B == 4) return f32_launch<B, 4, 8>(p, X, n, ldx, Y, ldy, s);
    return f32_launch<B, B == 4 ? 4 : 8, 8>(p, X, n, ldx, Y, ldy, s);
}

}  // namespace

cudaError_t launch_f32(const spmm_plan *p, const void *X, int64_t n, int64_t ldx, void *Y,
                       int64_t ldy, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (p->b == 4) return f32_dispatch<4>(p, X, n, ldx, Y, ldy, s);
    if (p->b == 8) return f32_dispatch<8>(p, X, n, ldx, Y, ldy, s);
    return f32_dispatch<16>(p, X, n, ldx, Y, ldy, s);
}

}  // namespace spmm
