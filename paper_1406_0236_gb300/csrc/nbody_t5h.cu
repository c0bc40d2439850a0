// FP32 inter-body sum y = B sigma (Sec. 3.3, Eq. (nystromnaive)) for several right-hand
// sides, the contraction over sources on the tensor cores (tcgen05, FP16 operands in a
// three-term split, FP32 accumulators), the pair kernels going from the registers that
// form them straight into tensor memory.
//
// A CTA of 256 threads owns 128 targets of one TargetBlock (4 CTAs per block) and RC = 16
// or 32 right-hand sides; two threads per target.  Sources come in tiles of 32 of one body.
// For every tile
//   * its geometry (structure of arrays) and the densities' operand images, both laid out in
//     global memory beforehand (t5h_source_kernel once per geometry, t5h_density_kernel once
//     per call), arrive by bulk copy into one of two shared-memory stages;
//   * each thread forms the kernels of its target with 16 of the sources, two per f32x2
//     instruction, G' = (n~.d) P + b - i a as in nbody32_sym_kernel (19 lane operations per
//     pair, 3 on the transcendental unit), cuts Re G' and -Im G' into an FP16 high part (11
//     leading bits) and the rounded rest, and stores the four parts as columns of its own
//     row of tensor memory (tcgen05.st): the A operands of the MMAs, which shared memory
//     never sees;
//   * one thread issues 12 MMAs (M = 128, N = 2 RC, K = 16; high x low, low x high and last high x
//     high, for Re G' x [Re s | Im s] and -Im G' x [Im s | -Re s]) and commits them.  The accumulator
//     is truncated at every MMA: with the small products first four of the twelve are at its full
//     size.  Error at 8,200 unknowns, k = 2, R = 12: 6.4e-7 with the three products of a factor in
//     turn, 5.0e-7 now, 5.3e-7 in FP32 multiply-adds;
//   * the warps read the accumulator (started from zero in every tile: chained tensor-core
//     sums are not rounded to nearest and drift) and add it, times the tile's scale, to FP32
//     sums in registers.
// One block barrier per tile; three CTAs per SM (128 columns of tensor memory each) overlap
// one another's barriers, MMAs and reads.
//
// FP16's range: G' is scaled by the power of two that brings its bound at the smallest
// distance between two bodies (t5h_range_kernel, once per geometry) to 2^15, the densities by tile
// and right-hand side to 2^14, so that a value down to 2^-17 of the largest keeps 22 bits and no
// value overflows.  The tile's power of two, against the column's, goes with its images (one scale
// per column left 2^-38 of the column's largest value to a body whose densities are small, and
// the rows of the others nothing else to sum: relative error 4e-4 there at 1e-8; now 1e-6, for
// 905 -> 915 to 930 us at 29,280 unknowns, R = 16).  Geometries whose kernels span more than FP16 (or k, eta
// outside sym_scaled) keep the TF32 form (nbody_tc5.cu).
//
// Bound by the transcendental unit (3 operations per ordered pair: 0.39 ms at 29,280
// unknowns) and issue (29 instructions per pair, a packed one counting twice at dispatch).  Against the TF32
// form of nbody_tc5.cu, whose operands went through shared memory: 29,280 unknowns, R = 16 1.74 ->
// 0.91 ms (error 3.1e-6 -> 2.9e-6); R = 32 1.08 ms; 64,640 unknowns, R = 16 4.5, R = 64 10.4 ms;
// 2,230,272 unknowns, R = 16 9.96 -> 5.59 s.  Two, three and four CTAs per SM measured 5.53, 4.69 and
// 4.74 ms at 64,640, R = 16 (before the transposed images); forming part of the next tile while the
// MMAs run gained nothing.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "f32x2.cuh"
#include "hzb_internal.h"
#include "kernel_math.cuh"
#include "sigma_scale.cuh"
#include "tcgen05.cuh"

namespace hzb {

static const int TH_M = 128;                           // targets per CTA = MMA M = lanes of tensor memory
static const int TH_S = 32;                            // sources per tile
static const int TH_THREADS = 256;
static const int TH_SRC = 6 * TH_S;                    // floats of a tile's geometry: x, y, z, nx, ny, nz
static const int TH_COLS = 128;                        // tensor-memory columns: A 64, D 2 RC
static const int TH_A = 0, TH_D = 64;                  // first columns
static const int TH_ATILE = TH_S / 2;                  // columns of one A part (two FP16 per column)
// Exponents below the column's largest value at which a tile's scale stops: 2^-100 of it times a sum
// of 2^-40 (in units of 2^29 and more) is still in FP32's range
static const int TH_LOW = 100;

__host__ __device__ constexpr int th_bytes(int rc) { return 2 * 2 * rc * 128; }   // B images of a tile: 2 x 2 RC rows
__host__ __device__ constexpr int th_image(int rc) { return th_bytes(rc) + 4 * rc; }          // and its scales
__host__ __device__ constexpr int th_stage(int rc) { return th_bytes(rc) + 1024; }
// two stages and the scales of four tiles: a stage is refilled while slower warps still read the
// scales of the tile that left it
__host__ __device__ constexpr int th_smem(int rc) { return 2 * th_stage(rc) + 4 * 4 * rc + 1024; }
static_assert(TH_SRC * 4 <= 1024, "geometry of a tile in its stage");

// kind::f16 with FP16 A and B, FP32 D
__host__ __device__ constexpr uint32_t th_idesc(int n)
{
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TH_M >> 4) << 24);
}

// D += A B^T with A in tensor memory
__device__ __forceinline__ void th_mma(uint32_t d, uint32_t a, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
        "r"(a), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void th_st4(uint32_t taddr, const uint32_t *r)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
}

template <int NN>
__device__ __forceinline__ void th_stn(uint32_t taddr, const uint32_t *r)
{
    if (NN == 4) th_st4(taddr, r);
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(taddr), "r"(r[0]), "r"(r[1])
                     : "memory");
}

__device__ __forceinline__ void th_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

// acc += f x NC columns of this warp's lanes
template <int NC>
__device__ __forceinline__ void th_add(uint32_t taddr, const float *f, float *acc)
{
#pragma unroll
    for (int q0 = 0; q0 < NC; q0 += 16) {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
            "%15}, [%16];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr + q0));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int q = 0; q < 16; q += 4) {
            const float4 s = *reinterpret_cast<const float4 *>(f + q0 + q);
            acc[q0 + q] = fmaf(__uint_as_float(r[q]), s.x, acc[q0 + q]);
            acc[q0 + q + 1] = fmaf(__uint_as_float(r[q + 1]), s.y, acc[q0 + q + 1]);
            acc[q0 + q + 2] = fmaf(__uint_as_float(r[q + 2]), s.z, acc[q0 + q + 2]);
            acc[q0 + q + 3] = fmaf(__uint_as_float(r[q + 3]), s.w, acc[q0 + q + 3]);
        }
    }
}

// FP16 parts of a packed pair: the 11 leading bits, and the rest rounded to 11 bits
__device__ __forceinline__ void th_cut(f2x x, uint32_t &hi, uint32_t &lo)
{
    float a, b;
    f2_unpack(x, a, b);
    const float ha = __uint_as_float(__float_as_uint(a) & 0xFFFFE000u);
    const float hb = __uint_as_float(__float_as_uint(b) & 0xFFFFE000u);
    const f2x l = f2_sub(x, f2_pack(ha, hb));
    f2_unpack(l, a, b);
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(hb), "f"(ha));
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(b), "f"(a));
}

template <int RC>
__global__ void __launch_bounds__(TH_THREADS, 3)
nbody_t5h_kernel(const TargetBlock *__restrict__ blocks, const int2 *__restrict__ own_tiles, int ntiles, int chunk,
                 int R, const float4 *__restrict__ pos, const float *__restrict__ src,
                 const unsigned char *__restrict__ img, float gscale, float2 *__restrict__ out, size_t split_stride,
                 int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char th_raw[];
    __shared__ uint32_t s_taddr;
    __shared__ __align__(8) unsigned long long s_bar[3];       // full[2], mma
    __shared__ int s_forced;                                   // host-set flag: take the timeout exit
    const TargetBlock tb = blocks[blockIdx.x >> 2];
    const int sub = blockIdx.x & 3;
    if (sub * TH_M >= tb.count) return;                        // whole CTA past the block's end
    const uint32_t base = ((uint32_t)__cvta_generic_to_shared(th_raw) + 1023u) & ~1023u;
    unsigned char *const gbase = th_raw + (base - (uint32_t)__cvta_generic_to_shared(th_raw));
    const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(&s_bar[0]);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quarter = warp & 3, half = warp >> 2;            // rows 32 quarter + lane; sources 16 half ..
    const int row = 32 * quarter + lane, t = sub * TH_M + row;
    constexpr int STAGE = th_stage(RC), BYTES = th_bytes(RC);
    // sources formed at a time, in fours: as many as 80 registers hold (three CTAs per SM)
    constexpr int G = RC == 16 ? 2 : 1;
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s_taddr);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(TH_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < 3; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar0 + 8 * q), "r"(1) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        s_forced = *(volatile int *)err < 0 ? 1 : 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_taddr;
    const uint32_t arow = tmem + ((uint32_t)(32 * quarter) << 16) + TH_A + 8 * half;
    const uint32_t drow = tmem + ((uint32_t)(32 * quarter) << 16) + TH_D + RC * half;

    f2x tx = f2_splat(1e5f + row), ty = f2_splat(1e5f), tz = ty;
    if (t < tb.count) {
        const float4 p = pos[tb.start + t];
        tx = f2_splat(p.x); ty = f2_splat(p.y); tz = f2_splat(p.z);
    }
    const f2x gs = f2_splat(gscale);
    float acc[RC];
#pragma unroll
    for (int q = 0; q < RC; ++q) acc[q] = 0.f;
    // the tiles of the other bodies, counted without the own body's [own.x, own.y)
    const int2 own = own_tiles[blockIdx.x >> 2];
    const int nown = own.y - own.x;
    const int i0 = blockIdx.z * chunk, i1 = min(ntiles - nown, i0 + chunk);
    // an injected fault ends the CTA before any copy or MMA is issued
    const int n = s_forced ? 0 : max(0, i1 - i0);
    auto issue = [&](int i) {
        const int q = i0 + i, tile = q < own.x ? q : q + nown;
        const uint32_t st = base + (uint32_t)((i & 1) * STAGE), mb = bar0 + 8 * (i & 1);
        const unsigned char *const im = img + ((size_t)tile * gridDim.y + blockIdx.y) * th_image(RC);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(BYTES + TH_SRC * 4 + 4 * RC)
                     : "memory");
        th_copy(st, im, BYTES, mb);
        th_copy(st + BYTES, src + (size_t)tile * TH_SRC, TH_SRC * 4, mb);
        th_copy(base + 2 * STAGE + (i & 3) * 4 * RC, im + BYTES, 4 * RC, mb);
    };
    if (tid == 0) {
        if (n > 0) issue(0);
        if (n > 1) issue(1);
    }
    int issued = min(n, 2), done = 0;                          // copies issued and seen complete (thread 0's view)
    bool ok = true, mma_ok = true;
    int last = 0;
    auto arrived = [&](int i) {
        if (t5_wait(bar0 + 8 * (i & 1), (uint32_t)((i >> 1) & 1))) done = i + 1;
        else ok = false;
    };
    // kernels of the thread's target with 4 G sources (group g of its 16) of tile i: 2 G columns of
    // each of the four parts
    auto form = [&](int i, int g, uint32_t (&part)[4][2 * G]) {
        const float *S = reinterpret_cast<const float *>(gbase + (i & 1) * STAGE + BYTES) + 16 * half + 4 * G * g;
#pragma unroll
        for (int v = 0; v < G; ++v) {
            ulonglong2 c[6];
#pragma unroll
            for (int a = 0; a < 6; ++a) c[a] = *reinterpret_cast<const ulonglong2 *>(S + 4 * v + a * TH_S);
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const f2x dx = f2_sub(tx, w ? c[0].y : c[0].x), dy = f2_sub(ty, w ? c[1].y : c[1].x),
                          dz = f2_sub(tz, w ? c[2].y : c[2].x);
                const f2x r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
                float ra, rb, sa, ca, sb, cb;
                f2_unpack(r2, ra, rb);
                const f2x ir = f2_pack(rsqrtf(ra), rsqrtf(rb));
                f2_unpack(f2_mul(r2, ir), ra, rb);
                __sincosf(ra, &sa, &ca);
                __sincosf(rb, &sb, &cb);
                const f2x is = f2_mul(ir, gs);
                const f2x ea = f2_mul(f2_pack(ca, cb), is), eb = f2_mul(f2_pack(sa, sb), is);
                const f2x X = f2_mul(ir, f2_fma(w ? c[3].y : c[3].x, dx,
                                                f2_fma(w ? c[4].y : c[4].x, dy, f2_mul(w ? c[5].y : c[5].x, dz))));
                const f2x gr = f2_fma(X, f2_fma(ea, ir, eb), eb), gn = f2_fma(X, f2_fma(f2_neg(eb), ir, ea), ea);
                th_cut(gr, part[0][2 * v + w], part[1][2 * v + w]);
                th_cut(gn, part[2][2 * v + w], part[3][2 * v + w]);
            }
        }
    };
    auto store = [&](int g, const uint32_t (&part)[4][2 * G]) {
#pragma unroll
        for (int q = 0; q < 4; ++q) th_stn<2 * G>(arow + q * TH_ATILE + 2 * G * g, part[q]);
    };
    for (int i = 0; i < n; ++i) {
        arrived(i);
#pragma unroll 1
        for (int g = 0; g < 4 / G; ++g) {
            uint32_t part[4][2 * G];
            form(i, g, part);
            store(g, part);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        // every thread's columns are in place and its reads of D and of the stage's geometry done;
        // a wait that ran out anywhere ends the loop for all
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        if (warp == 0 && t5_elect()) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t desc = t5_desc(base + (uint32_t)((i & 1) * STAGE));
#pragma unroll
            for (int term = 0; term < 3; ++term)               // high x low, low x high, then high x high
#pragma unroll
                for (int z = 0; z < 2; ++z)                    // Re G' x B1, -Im G' x B2
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {
                        const uint32_t a = tmem + TH_A + (2 * z + (term == 1 ? 1 : 0)) * TH_ATILE + 8 * ks;
                        const uint64_t b = desc + ((z * (BYTES / 2) + 32 * ks + (term == 0 ? 64 : 0)) >> 4);
                        th_mma(tmem + TH_D, a, b, th_idesc(2 * RC), (term | z | ks) ? 1u : 0u);
                    }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar0 + 16)
                         : "memory");
        }
        mma_ok = t5_wait(bar0 + 16, (uint32_t)(i & 1));
        ok &= mma_ok;
        last = i;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (tid == 0 && ok && i + 2 < n) {                     // the stage is free: MMAs done, geometry read
            issue(i + 2);
            issued = i + 3;
        }
        th_add<RC>(drow, reinterpret_cast<const float *>(gbase + 2 * STAGE) + (i & 3) * RC, acc);
    }
    if (tid == 0) {                                            // after a timeout: what is in flight, once more
        if (!mma_ok) t5_wait(bar0 + 16, (uint32_t)(last & 1));
        for (int i = done; i < issued; ++i) t5_wait(bar0 + 8 * (i & 1), (uint32_t)((i >> 1) & 1));
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    const bool failed = __syncthreads_or(!ok) || s_forced;
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TH_COLS) : "memory");
    if (failed && tid == 0) atomicExch(err, 1);
    if (t >= tb.count) return;
    // columns RC half ..: real parts (half 0) or imaginary parts
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const int rr = blockIdx.y * RC + r;
        if (rr >= R) break;
        float *o = reinterpret_cast<float *>(out + blockIdx.z * split_stride + (size_t)(tb.start + t) * R + rr);
        o[half] = failed ? __int_as_float(0x7fc00000) : acc[r];
    }
}

// ---------------------------------------------------------------- operand images

// geometry of the tiles: positions times ps about o, normals times ns; padding sources far away
__global__ void t5h_source_kernel(int ntiles, const int2 *__restrict__ tiles, const double4 *__restrict__ pos,
                                  const double4 *__restrict__ nrm, double3 o, double ps, double ns,
                                  float *__restrict__ src, float4 *__restrict__ ball)
{
    const int tile = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (tile >= ntiles) return;
    const int2 tl = tiles[tile];
    const bool have = lane < tl.y;
    float v[6] = {-1e5f - lane, -1e5f, -1e5f, 0.f, 0.f, 0.f};
    if (have) {
        const double4 p = pos[tl.x + lane], n = nrm[tl.x + lane];
        v[0] = (float)((p.x - o.x) * ps); v[1] = (float)((p.y - o.y) * ps); v[2] = (float)((p.z - o.z) * ps);
        v[3] = (float)(n.x * ns); v[4] = (float)(n.y * ns); v[5] = (float)(n.z * ns);
    }
#pragma unroll
    for (int a = 0; a < 6; ++a) src[(size_t)tile * TH_SRC + a * TH_S + lane] = v[a];
    // a ball about the tile, for the range
    float c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float s = have ? v[a] : 0.f;
        for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
        c[a] = s / tl.y;
    }
    const float dx = v[0] - c[0], dy = v[1] - c[1], dz = v[2] - c[2];
    float r = have ? sqrtf(dx * dx + dy * dy + dz * dz) : 0.f;
    for (int q = 16; q > 0; q >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, q));
    if (lane == 0) ball[tile] = make_float4(c[0], c[1], c[2], r * 1.0001f);
}

// smallest distance between nodes of different bodies (range[0], bits; in the scaled lengths, a
// lower bound within a factor of two: balls first, node by node where the balls are no use)
// and an upper bound of the largest (range[1]).  One warp per tile i against the tiles of
// later bodies.
__global__ void t5h_range_kernel(int ntiles, const int2 *__restrict__ tiles, const int2 *__restrict__ body_end,
                                 const float *__restrict__ src, const float4 *__restrict__ ball, int *__restrict__ range)
{
    const int i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= ntiles) return;
    const float4 bi = ball[i];
    const float *si = src + (size_t)i * TH_SRC;
    float best = 3e38f, far = 0.f;
    for (int j0 = body_end[i].x; j0 < ntiles; j0 += 32) {
        const int j = j0 + lane;
        bool close = false;
        if (j < ntiles) {
            const float4 bj = ball[j];
            const float dx = bi.x - bj.x, dy = bi.y - bj.y, dz = bi.z - bj.z;
            const float d = sqrtf(dx * dx + dy * dy + dz * dz), b = d * 0.9999f - bi.w - bj.w;
            close = !(b >= 0.5f * d);
            if (!close) best = fminf(best, b);
            far = fmaxf(far, d * 1.0001f + bi.w + bj.w);
        }
        unsigned m = __ballot_sync(0xffffffffu, close);
        while (m) {
            const int j1 = j0 + __ffs(m) - 1;
            m &= m - 1;
            const float *sj = src + (size_t)j1 * TH_SRC;
            if (lane < tiles[j1].y)
                for (int q = 0; q < tiles[i].y; ++q) {
                    const float x = sj[lane] - si[q], y = sj[TH_S + lane] - si[TH_S + q],
                                z = sj[2 * TH_S + lane] - si[2 * TH_S + q];
                    best = fminf(best, 0.999f * sqrtf(x * x + y * y + z * z));
                }
        }
    }
    for (int q = 16; q > 0; q >>= 1) {
        best = fminf(best, __shfl_xor_sync(0xffffffffu, best, q));
        far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, q));
    }
    if (lane == 0) {
        atomicMin(&range[0], __float_as_int(fmaxf(best, 0.f)));
        atomicMax(&range[1], __float_as_int(far));
    }
}

// B images of every tile and chunk of RC right-hand sides, in the swizzled K-major layout the
// MMAs read: rows n < RC and n + RC of B1 = [Re s' ; Im s'] and B2 = [Im s' ; -Re s'], each row
// the high parts of the 32 sources, then the low parts; behind them the scales of the RC columns.
// s' = w sigma 2^(14 - e), e the exponent of the tile's largest value (at least the column's - TH_LOW);
// the scale 2^(e - the column's).  A warp takes eight columns, a lane one of them and eight sources.
__global__ void t5h_density_kernel(int ntiles, int R, int rc, int nchunk, const int2 *__restrict__ tiles,
                                   const double4 *__restrict__ pos, const double2 *__restrict__ sigma,
                                   const int *__restrict__ key, unsigned char *__restrict__ img)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int ncol = rc * nchunk;
    if (e >= (size_t)ntiles * ncol * 4) return;
    const int lane = threadIdx.x & 31, g = lane >> 3, per = ncol / 8;
    const int tile = (int)(e / 32 / per), col = (int)(e / 32 % per) * 8 + (lane & 7);
    const int2 tl = tiles[tile];
    const int top = col < R ? sigma_exponent(key[col]) : 0;
    double2 z[8];
    int big = 0;                                               // largest high word of the finite values
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int s = 8 * g + q;
        z[q] = make_double2(0.0, 0.0);
        if (s < tl.y && col < R) {
            const double wq = pos[tl.x + s].w;
            z[q] = sigma[(size_t)(tl.x + s) * R + col];
            z[q].x *= wq;
            z[q].y *= wq;
            const int hx = __double2hiint(z[q].x) & 0x7fffffff, hy = __double2hiint(z[q].y) & 0x7fffffff;
            big = max(big, max(hx < 0x7ff00000 ? hx : 0, hy < 0x7ff00000 ? hy : 0));
        }
    }
    big = max(big, __shfl_xor_sync(0xffffffffu, big, 8));
    big = max(big, __shfl_xor_sync(0xffffffffu, big, 16));
    const int own = min(top, max(top - TH_LOW, big ? sigma_exponent(big) : -960));
    const double sc = sigma_pow2(14 - own);
    uint32_t h[2][4], l[2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float v[2][2];
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            v[0][w] = (float)(z[2 * q + w].x * sc);
            v[1][w] = (float)(z[2 * q + w].y * sc);
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const __half2 hh = __floats2half2_rn(v[a][0], v[a][1]);
            const __half2 ll = __floats2half2_rn(v[a][0] - __low2float(hh), v[a][1] - __high2float(hh));
            h[a][q] = *reinterpret_cast<const uint32_t *>(&hh);
            l[a][q] = *reinterpret_cast<const uint32_t *>(&ll);
        }
    }
    const int n = col % rc, bytes = th_bytes(rc);
    unsigned char *b1 = img + ((size_t)tile * nchunk + col / rc) * th_image(rc), *b2 = b1 + bytes / 2;
    if (g == 0) reinterpret_cast<float *>(b1 + bytes)[n] = (float)sigma_pow2(own - top);
    const uint32_t neg = 0x80008000u;
    auto put = [&](unsigned char *b, int row, const uint32_t *hi, const uint32_t *lo, uint32_t flip) {
        *reinterpret_cast<uint4 *>(b + t5_chunk_off(row, g)) =
            make_uint4(hi[0] ^ flip, hi[1] ^ flip, hi[2] ^ flip, hi[3] ^ flip);
        *reinterpret_cast<uint4 *>(b + t5_chunk_off(row, g + 4)) =
            make_uint4(lo[0] ^ flip, lo[1] ^ flip, lo[2] ^ flip, lo[3] ^ flip);
    };
    put(b1, n, h[0], l[0], 0u);
    put(b1, n + rc, h[1], l[1], 0u);
    put(b2, n, h[1], l[1], 0u);
    put(b2, n + rc, h[0], l[0], neg);
}

// y = f 2^(exponent - 14) sum over the source chunks.  The FP32 partial sums are added by two-sums
// in FP32 (their error below FP64's rounding of y's own FP32 error): an FP64 addition and a
// conversion per value kept the FP64 pipe busy for most of the 61 us that 29,280 unknowns,
// 16 right-hand sides and 15 chunks took (now 19 us).
__device__ __forceinline__ void t5h_add(float &h, float &l, float v)
{
    const float s = __fadd_rn(h, v), b = __fsub_rn(s, h);
    l += __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(v, b));
    h = s;
}
__global__ void t5h_reduce_kernel(size_t n, int R, int nsplit, double f, const int *__restrict__ key,
                                  const float2 *__restrict__ part, double2 *__restrict__ y)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    float xh = 0.f, xl = 0.f, yh = 0.f, yl = 0.f;
#pragma unroll 4
    for (int s = 0; s < nsplit; ++s) {
        const float2 v = part[s * n + e];
        t5h_add(xh, xl, v.x);
        t5h_add(yh, yl, v.y);
    }
    const double sc = f * sigma_pow2(sigma_exponent(key[e % R]) - 14);
    y[e] = make_double2(((double)xh + (double)xl) * sc, ((double)yh + (double)yl) * sc);
}

// ---------------------------------------------------------------- host

// Tiles, their geometry and the range of the kernel, once per geometry.
hzb_status ensure_t5h(hzb_ctx *c)
{
    if (c->t5h_state) return HZB_OK;
    if (c->capturing) return fail(c, HZB_ESTATE, "tiles not built before capture");
    if (!sym_scaled(c)) {
        c->t5h_state = -1;
        return HZB_OK;
    }
    hzb_status st0 = ensure_sym32(c);                          // the targets' scaled positions
    if (st0) return st0;
    std::vector<TargetBlock> tb(c->n_tblocks);
    if (check_cuda(c, cudaMemcpyAsync(tb.data(), c->tblocks.ptr, tb.size() * sizeof(TargetBlock),
                                      cudaMemcpyDeviceToHost, c->stream), "copy blocks") ||
        check_cuda(c, cudaStreamSynchronize(c->stream), "copy blocks"))
        return HZB_ECUDA;
    // one buffer: the tiles, the blocks' own tiles, the end of each tile's body, the range, the tiles' words
    std::vector<int2> tiles, own(tb.size()), end;
    std::vector<int> word;
    int nbodies = 0;
    for (size_t b = 0; b < tb.size(); ++b) {
        if (b == 0 || tb[b].excl_lo != tb[b - 1].excl_lo) {    // a new body: its nodes are one range
            const int first = (int)tiles.size();
            for (int s = tb[b].excl_lo; s < tb[b].excl_hi; s += TH_S) {
                const int count = std::min(TH_S, tb[b].excl_hi - s);
                word.push_back(t5h_tile_word(nbodies, ((int)tiles.size() - first) & 1, count));
                tiles.push_back(make_int2(s, count));
            }
            ++nbodies;
            end.resize(tiles.size(), make_int2((int)tiles.size(), 0));
            own[b] = make_int2(first, (int)tiles.size());
        } else {
            own[b] = own[b - 1];
        }
    }
    const int nt = (int)tiles.size();
    tiles.insert(tiles.end(), own.begin(), own.end());
    tiles.insert(tiles.end(), end.begin(), end.end());
    tiles.push_back(make_int2(0x7f7fffff, 0));
    const size_t words = tiles.size();
    if (nt & 1) word.push_back(0);
    for (int q = 0; q < nt; q += 2) tiles.push_back(make_int2(word[q], word[q + 1]));
    if (check_cuda(c, c->t5h_tiles.ensure(tiles.size()), "alloc tiles") ||
        check_cuda(c, c->t5h_src.ensure((size_t)nt * (TH_SRC + 4)), "alloc tiles"))
        return HZB_ENOMEM;
    float4 *ball = reinterpret_cast<float4 *>(c->t5h_src.ptr + (size_t)nt * TH_SRC);
    int2 *const end_dev = c->t5h_tiles.ptr + nt + own.size();
    int *const range_dev = reinterpret_cast<int *>(end_dev + nt);
    if (check_cuda(c, cudaMemcpyAsync(c->t5h_tiles.ptr, tiles.data(), tiles.size() * sizeof(int2), cudaMemcpyHostToDevice,
                                      c->stream), "copy tiles"))
        return HZB_ECUDA;
    t5h_source_kernel<<<(nt + 7) / 8, 256, 0, c->stream>>>(
        nt, c->t5h_tiles.ptr, c->pos64.ptr, c->nrm64.ptr, make_double3(c->center[0], c->center[1], c->center[2]), c->k,
        c->k / c->eta, c->t5h_src.ptr, ball);
    t5h_range_kernel<<<(nt + 7) / 8, 256, 0, c->stream>>>(nt, c->t5h_tiles.ptr, end_dev, c->t5h_src.ptr, ball, range_dev);
    float range[2];
    if (check_cuda(c, cudaGetLastError(), "tiles") ||
        check_cuda(c, cudaMemcpyAsync(range, range_dev, sizeof(range), cudaMemcpyDeviceToHost, c->stream), "copy range") ||
        check_cuda(c, cudaStreamSynchronize(c->stream), "tiles"))
        return HZB_ECUDA;
    const double g = range[0], diam = range[1];
    // |G'| <= u (1 + (k / |eta|) (1 + u)), u = 1 / (k r); the smallest is about u at the diameter
    c->t5h_ntiles = nt;
    c->t5h_nbodies = nbodies;
    c->t5h_words = reinterpret_cast<const int *>(c->t5h_tiles.ptr + words);
    c->t5h_ctas = 0;
    for (const TargetBlock &t : tb) c->t5h_ctas += (t.count + TH_M - 1) / TH_M;
    c->t5h_most = 1;                                           // tiles of the other bodies, at most
    for (const int2 &o : own) c->t5h_most = std::max(c->t5h_most, nt - (o.y - o.x));
    double sum = 0.0;                                          // and their mean over the CTAs
    for (size_t b = 0; b < tb.size(); ++b) sum += (double)((tb[b].count + TH_M - 1) / TH_M) * (nt - (own[b].y - own[b].x));
    c->t5h_mean = c->t5h_ctas ? sum / c->t5h_ctas : 1.0;
    // |G| <= u (u + 1 + |eta| / k): its bounds at the smallest and the largest distance (nbody_dfx.cu)
    const double q = 1.0 + std::fabs(c->eta) / c->k;
    c->t5h_span = g > 0.0 && diam > 0.0 && diam < 9e4 ? (1.0 / g) * (1.0 / g + q) / ((1.0 / diam) * (1.0 / diam + q)) : 0.0;
    const double u = 1.0 / g, bound = u * (1.0 + (c->k / std::fabs(c->eta)) * (1.0 + u)) * 1.001;
    c->t5h_state = -1;
    if (std::isfinite(bound) && g > 0.0 && diam > 0.0 && diam < 9e4 && bound * diam < 262144.0) {
        int e;
        std::frexp(bound, &e);                                 // bound < 2^e
        if (e > -100 && e < 100) {
            c->t5h_scale = std::ldexp(1.0, 15 - e);
            c->t5h_state = 1;
        }
    }
    return HZB_OK;
}

// whether the context's geometry, k and eta suit this form (-1 in *st: an error)
bool t5h_usable(hzb_ctx *c, hzb_status *st)
{
    *st = ensure_t5h(c);
    return !*st && c->t5h_state > 0;
}

hzb_status interbody_t5h(hzb_ctx *c, int R, const double2 *sigma, double2 *y)
{
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->opt.device);
    const int rc = R <= 16 ? 16 : 32, nchunk = (R + rc - 1) / rc, nt = c->t5h_ntiles;
    const int most = c->t5h_most;
    // Source chunks: the number that gives the shortest sum of the kernel's time (2.5 pairs per
    // clock and SM, over the fill of its last wave) and of the partial sums' (8 us per 10^6
    // values written and read), at least eight tiles to each.
    const long long ctas = (long long)c->t5h_ctas * nchunk, places = 3LL * sms;
    const double full = (double)ctas * TH_M * TH_S * most / (2.5 * 2.0e3 * sms), part = 8e-6 * (double)c->N * R;
    int nsplit = 1;
    double best = 1e300;
    for (int ns = 1; ns <= std::max(1, std::min(64, most / 8)); ++ns) {
        const double waves = (double)(ns * ctas) / places, t = full * std::ceil(waves) / waves + part * ns;
        if (t < best) { best = t; nsplit = ns; }
    }
    const int chunk = (most + nsplit - 1) / nsplit;
    nsplit = (most + chunk - 1) / chunk;
    const size_t n = (size_t)c->N * R;
    if (check_cuda(c, c->nb_part32.ensure(n * nsplit), "alloc partial sums") ||
        check_cuda(c, c->t5h_img.ensure((size_t)nt * nchunk * th_image(rc)), "alloc operand images") ||
        check_cuda(c, c->dlkey.ensure(R), "alloc scales"))
        return HZB_ENOMEM;
    hzb_status st = tc_flag_begin(c, FAULT_TIMEOUT);
    if (st) return st;
    const int smem = th_smem(rc);                              // below the 48 KB that need no attribute
    static_assert(th_smem(32) <= 48 * 1024, "dynamic shared memory");
    c->interbody_calls++;
    const int slot = prof_begin(c, 1);
    if ((st = sigma_keys(c, R, sigma, 1.0, 1, c->dlkey.ptr))) return st;
    const size_t ne = (size_t)nt * rc * nchunk * 4;
    t5h_density_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, c->stream>>>(nt, R, rc, nchunk, c->t5h_tiles.ptr,
                                                                          c->pos64.ptr, sigma, c->dlkey.ptr,
                                                                          c->t5h_img.ptr);
    const dim3 grid((unsigned)c->n_tblocks * 4, nchunk, nsplit);
    auto launch = [&](auto kern) {
        kern<<<grid, TH_THREADS, smem, c->stream>>>(c->tblocks.ptr, c->t5h_tiles.ptr + nt, nt, chunk, R,
                                                    c->symn.ptr, c->t5h_src.ptr, c->t5h_img.ptr, (float)c->t5h_scale,
                                                    c->nb_part32.ptr, n, c->kerr.ptr);
    };
    if (rc == 16) launch(nbody_t5h_kernel<16>);
    else launch(nbody_t5h_kernel<32>);
    t5h_reduce_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(
        n, R, nsplit, c->k * c->eta * HZB_INV4PI / c->t5h_scale, c->dlkey.ptr, c->nb_part32.ptr, y);
    c->launches += 3;
    cudaError_t e = cudaGetLastError();
    prof_end(c, slot);
    if (check_cuda(c, e, "nbody_t5h_kernel")) return HZB_ECUDA;
    // on automatic fewer than 16 right-hand sides are queued like the CUDA cores' sums
    return tc_flag_end(c, "nbody_t5h_kernel", R >= 16 || c->nbody_engine >= 0);
}

}  // namespace hzb
