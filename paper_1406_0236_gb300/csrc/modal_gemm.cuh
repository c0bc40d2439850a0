// Batched complex GEMM C[p] = A[p] B[p] of the block-diagonal inverse on the CUDA cores, for
// FP64, FP32 and double-float values: A n x n, B and C n x nc, row-major, one matrix of each
// per azimuthal mode p.
//
// A warp owns TM rows; its lanes are LC columns times 32 / LC shares of the k sum, added by
// shuffles at the end, so that panels of 2, 4, 8, ... columns (one or two right-hand sides on
// one or two bodies) keep every lane busy and the k chain short.  Rows beyond n cost nothing
// (a warp without a row leaves the loop), and a block is only WARPS x TM rows high: the grid has
// several blocks per SM at N_G = 100 and 21 modes.  Tiles are staged by cp.async, KC of the n
// terms at a time: all of them when they fit in 40 KB, which is one wait for the whole product.
//
// Whole D^{-1} before -> after, two bodies of N_G = 100, 21 modes (us): FP64, R = 1, 4, 64:
// 127 -> 30, 148 -> 91, 1394 -> 567; double-float 59 -> 20, 66 -> 27, 327 -> 187; FP32, R = 1:
// 25 -> 18 (DFTs included on both sides, theirs folded meanwhile).  Tiles of the wide form
// (rows x columns to a lane), double-float, R = 64: 2 x 1 187, 1 x 1 188, 1 x 2 183, 2 x 2 187, 4 x 1
// 212; at R = 8 2 x 1 44, 1 x 2 55, 2 x 2 58.  FP64 is bound by its pipe (4 FMAs per term).
#pragma once

#include <algorithm>
#include <cuda_runtime.h>

#include "lean_df.cuh"

namespace hzb {

// the arithmetic of one element type: a complex accumulator, acc += a b, sums over lanes
template <typename E> struct ComplexAcc;

template <typename T, typename C>
struct ComplexAccPlain {
    T x, y;
    __device__ __forceinline__ ComplexAccPlain() : x((T)0), y((T)0) {}
    __device__ __forceinline__ void mac(C a, C b)
    {
        x += a.x * b.x;
        y += a.x * b.y;
        x -= a.y * b.y;
        y += a.y * b.x;
    }
    __device__ __forceinline__ void settle() {}
    __device__ __forceinline__ void add_lane(int m)
    {
        x += __shfl_xor_sync(0xffffffffu, x, m);
        y += __shfl_xor_sync(0xffffffffu, y, m);
    }
    __device__ __forceinline__ C value() const
    {
        C v;
        v.x = x;
        v.y = y;
        return v;
    }
};
template <> struct ComplexAcc<double2> : ComplexAccPlain<double, double2> {};
template <> struct ComplexAcc<float2> : ComplexAccPlain<float, float2> {};
template <> struct ComplexAcc<float4> {
    lean::dd x = {0.f, 0.f}, y = {0.f, 0.f};
    __device__ __forceinline__ void mac(float4 a, float4 b) { lean::cmac(x, y, a, b); }
    __device__ __forceinline__ void settle()
    {
        x = lean::norm(x);
        y = lean::norm(y);
    }
    __device__ __forceinline__ void add_lane(int m)
    {
        const lean::dd u = {__shfl_xor_sync(0xffffffffu, x.h, m), __shfl_xor_sync(0xffffffffu, x.l, m)};
        const lean::dd v = {__shfl_xor_sync(0xffffffffu, y.h, m), __shfl_xor_sync(0xffffffffu, y.l, m)};
        x = lean::norm(lean::add(x, u));
        y = lean::norm(lean::add(y, v));
    }
    __device__ __forceinline__ float4 value() const { return make_float4(x.h, x.l, y.h, y.l); }
};

template <typename E>
__device__ __forceinline__ void modal_stage(E *dst, const E *src, bool in)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = in ? (int)sizeof(E) : 0;                 // 0: the element is filled with zeros
    if (sizeof(E) == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes));
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(bytes));
}

template <typename E, int WARPS, int LC, int TM, int TN>
__global__ void __launch_bounds__(32 * WARPS)
modal_gemm_kernel(int n, int nc, int KC, const E *__restrict__ A, const E *__restrict__ B, E *__restrict__ C)
{
    constexpr int KQ = 32 / LC, BM = WARPS * TM, BN = LC * TN;
    extern __shared__ __align__(16) unsigned char modal_smem[];
    E *As = reinterpret_cast<E *>(modal_smem), *Bs = As + (size_t)BM * KC;    // BM x KC, KC x BN
    const int p = blockIdx.z, row0 = blockIdx.y * BM, col0 = blockIdx.x * BN;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, lc = lane % LC, kq = lane / LC;
    const E *Ap = A + (size_t)p * n * n, *Bp = B + (size_t)p * n * nc;
    ComplexAcc<E> acc[TM][TN];
    for (int k0 = 0; k0 < n; k0 += KC) {
        const int kc = min(KC, n - k0), iters = (kc + KQ - 1) / KQ;
        if (k0) __syncthreads();
        for (int r = w; r < BM && row0 + r < n; r += WARPS)
            for (int k = lane; k < iters * KQ; k += 32)
                modal_stage(As + r * KC + k, Ap + (size_t)(row0 + r) * n + (k < kc ? k0 + k : 0), k < kc);
        for (int e = tid; e < iters * KQ * BN; e += 32 * WARPS) {
            const int k = e / BN, col = col0 + e % BN;
            const bool in = k < kc && col < nc;
            modal_stage(Bs + e, in ? Bp + (size_t)(k0 + k) * nc + col : Bp, in);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (row0 + w >= n) continue;                           // (a later row of the warp may be stale, never stored)
        for (int i0 = 0; i0 < iters; i0 += 16) {
            const int i1 = min(i0 + 16, iters);
#pragma unroll 4
            for (int i = i0; i < i1; ++i) {
                const int k = i * KQ + kq;
                E b[TN];
#pragma unroll
                for (int q = 0; q < TN; ++q) b[q] = Bs[k * BN + lc + LC * q];
#pragma unroll
                for (int t = 0; t < TM; ++t) {
                    const E a = As[(w + t * WARPS) * KC + k];
#pragma unroll
                    for (int q = 0; q < TN; ++q) acc[t][q].mac(a, b[q]);
                }
            }
#pragma unroll
            for (int t = 0; t < TM; ++t)
#pragma unroll
                for (int q = 0; q < TN; ++q) acc[t][q].settle();
        }
    }
#pragma unroll
    for (int t = 0; t < TM; ++t) {
        const int row = row0 + w + t * WARPS;
#pragma unroll
        for (int q = 0; q < TN; ++q) {
#pragma unroll
            for (int m = LC; m < 32; m *= 2) acc[t][q].add_lane(m);
            const int col = col0 + lc + LC * q;
            if (kq == 0 && row < n && col < nc) C[((size_t)p * n + row) * nc + col] = acc[t][q].value();
        }
    }
}

// terms of the k sum staged at a time: a multiple of 32, or all n of them (rounded up to KQ)
// when that fits in 40 KB; wide tiles at most 64
template <typename E, int WARPS, int LC, int TM, int TN>
static void modal_gemm_launch(cudaStream_t st, int n, int nc, int modes, const E *A, const E *B, E *C)
{
    constexpr int KQ = 32 / LC, BM = WARPS * TM, BN = LC * TN, BYTES = (BM + BN) * (int)sizeof(E);
    constexpr int FIT = 40 * 1024 / BYTES / 32 * 32, MOST = TN * LC == 32 || TM > 1 ? std::min(FIT, 64) : FIT;
    static_assert(MOST >= 32, "a tile of 32 terms has to fit");
    const int kc = std::min((n + KQ - 1) / KQ * KQ, MOST);
    modal_gemm_kernel<E, WARPS, LC, TM, TN><<<dim3((nc + BN - 1) / BN, (n + BM - 1) / BM, modes), 32 * WARPS,
                                             (size_t)kc * BYTES, st>>>(n, nc, kc, A, B, C);
}

// TM, TN: the register tile of panels of more than 16 columns
template <typename E, int TM, int TN>
static void modal_gemm(cudaStream_t st, int n, int nc, int modes, const E *A, const E *B, E *C)
{
    if (nc <= 2) modal_gemm_launch<E, 4, 2, 1, 1>(st, n, nc, modes, A, B, C);
    else if (nc <= 4) modal_gemm_launch<E, 4, 4, 1, 1>(st, n, nc, modes, A, B, C);
    else if (nc <= 8) modal_gemm_launch<E, 4, 8, 1, 1>(st, n, nc, modes, A, B, C);
    else if (nc <= 16) modal_gemm_launch<E, 4, 16, 1, 1>(st, n, nc, modes, A, B, C);
    else modal_gemm_launch<E, 8, 32, TM, TN>(st, n, nc, modes, A, B, C);
}

}  // namespace hzb
