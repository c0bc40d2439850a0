// tcgen05 building blocks shared by the tensor-core kernels (5th-generation tensor
// cores: MMAs issued by one thread, operands in shared memory, accumulators in tensor
// memory): TF32 rounding, the 128-byte-swizzle K-major tile layout, shared-memory and
// instruction descriptors, the MMA, bounded mbarrier waits and tensor-memory loads.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace hzb {

__device__ __forceinline__ uint32_t t5_tf32(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// The same rounding (to nearest, ties away from zero, 10 stored mantissa bits) in two
// integer operations on the bit pattern: add half of the 13 dropped bits' range and
// clear them; equal to cvt.rna for every finite x, and for an infinity.  A NaN is lost: the
// hardware's 0x7fffffff becomes -0.  The conversion instruction has a fraction of the integer
// pipe's throughput, so the hot loops that split every pair kernel use this form; what a caller
// hands in (densities, panels of D^{-1}) goes through t5_tf32, which keeps a NaN.
__device__ __forceinline__ uint32_t t5_tf32i(float x) { return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u; }

// Byte offset of the 16-byte chunk c (4 TF32 values along K) of row `row` in a K-major
// tile with 128-byte rows and the 128-byte swizzle: 8-row atoms of 1024 bytes, chunk
// index XOR (row mod 8).
__device__ __forceinline__ uint32_t t5_chunk_off(int row, int c)
{
    return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((c ^ (row & 7)) << 4));
}

__device__ __forceinline__ void t5_st4(uint32_t saddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 1024-byte stride between
// 8-row groups, descriptor version 1.
__device__ __forceinline__ uint64_t t5_desc(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

// Instruction descriptor, kind::tf32: D FP32, A and B TF32, both K-major, N x M.
__host__ __device__ constexpr uint32_t t5_idesc(int n, int m = 128)
{
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void t5_mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate)
        : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ bool t5_elect()
{
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ bool t5_wait(uint32_t mbar, uint32_t parity)
{
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// Every wait gives up on its own lane's count of polls (and, where there is one, its own view of an
// abort flag).  A warp that goes on to warp-wide instructions (elect.sync, tcgen05.ld, __syncwarp)
// takes one answer for all its lanes: true where every lane's wait came through.
__device__ __forceinline__ bool t5_all(bool ok) { return __all_sync(0xffffffffu, ok); }

__device__ __forceinline__ void t5_ld32(uint32_t taddr, float *v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] += __uint_as_float(r[q]);
}

__device__ __forceinline__ void t5_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] += __uint_as_float(r[q]);
}

}  // namespace hzb
