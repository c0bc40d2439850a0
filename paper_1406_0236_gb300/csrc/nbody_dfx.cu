// Inter-body sum in double-float for several right-hand sides with the contraction on the tensor
// cores: pair kernels in lean double-float on the FP32 pipe (dfl_pair.cuh), the sums over sources
// as exact integer products of FP16 digits (tcgen05, FP32 accumulators).
//
// With G = E [X - i (kr X + eta')] (nbody_dfl.cu) and sigma' = w sigma c0 scaled below one per body
// and right-hand side, y_i = sum_j G_ij sigma'_j.  Each real number is cut into DX_D = 6 digits of
// base 2^9: x = G 2^E with |x| < 2^8 (E from a bound of |G| over the CTA's pairs) and
// s = 2^8 sigma' are x = sum_a d_a 2^(-9 a) with integers |d_a| <= 2^8 + 4, exact in FP16.  The
// products of digits a + b = l add up, over two tiles of 32 sources and real and imaginary parts, to
// an integer of at most (l + 1) 2^23 in the accumulator of level l: exact in FP32 for l <= 1, and for
// l = 2, 3 unless nearly every digit is at its limit with one sign, when a unit (2^-18 of a product
// of the leading digits) is lost on a sum of 2^23 of them.  The levels 0 ... 5 (21 products) are
// kept; what is left out is below 2^-50 of the largest product, the digits' own cut 2^-53 of the
// largest kernel value.  After two tiles of one body the six levels enter 64-bit integers (unit 2^-32),
// shifted from that body's scale to the largest of those the targets sum, their own body's left out:
// no sum is rounded but there.  (One scale over all bodies left a body whose densities are 1e-8 of the
// largest 1e-8 of relative error on the others' rows; the shifts and the levels moved at a body's end
// cost 3 % at 8,200 unknowns, R = 64, and on three bodies of 9,008 unknowns, R = 8.)  The integers hold 256 tiles; a longer chunk
// adds them to y (or its partial sum) in FP64 that often, so that the number of chunks follows the SMs
// alone (with a chunk per 256 tiles 258,560 unknowns and R = 64 took 7.4 GB of partial sums, 2.2 million
// and R = 16 152 GB).
//
// Per CTA: 128 targets (the M of the MMA), RC right-hand sides (N = 2 RC columns: real and
// imaginary parts), a chunk of the source tiles.  Sixteen warps form kernels, four sources of each
// half tile for a thread's target (row): one 16-byte chunk (four sources, real and imaginary part) of
// each of the six digit images of A in shared memory (K-major, 64-byte swizzle).  A seventeenth
// warp issues the half tile's 42 MMAs when all have arrived and fetches the digit images of the
// densities (dfx_density_kernel, one 128-byte row per column and digit) and the sources' nodes two
// tiles ahead; the sixteen never wait for one another.  Before the first MMA of every second tile
// they move the levels into the 64-bit sums, which live in tensor memory too (columns 12 RC ..
// 16 RC).
//
// More than 32 right-hand sides (tensor memory holds the levels and sums of 32): two CTAs of a
// cluster take the same targets and sources with 32 right-hand sides each, form half of every tile
// each and send it to the other by one bulk copy (stores to the other CTA's shared memory by the
// forming warps took 4,900 cycles a tile, as long as the forming).  Then the 84 MMAs of a tile (about
// 60 cycles each: both operands come from shared memory) and the forming take about equally long.
//
// Bound by the issue of the pair kernels and digits, about 260 + 55 FP32 operations per pair and
// RC right-hand sides (77 % of the issue slots at RC = 8); the one-directional kernel of
// nbody_dfl.cu spends another 28 slots per pair and right-hand side on the sums.  Against it, and
// the error of each against 64 bits:
//   29,280 unknowns, k = 6:  R = 4  8.70 -> 7.36 ms;  R = 8  10.9 -> 7.4;  R = 16  16.7 -> 7.7;
//                            R = 64  61.1 -> 12.3 ms, 1.2e-13 -> 1.1e-13
//   8,200 unknowns, k = 2:   R = 8  0.66 -> 0.47 ms;  R = 64  3.74 -> 0.78 ms, 5.6e-14 -> 3.4e-14
//   2,230,272 unknowns, k = 6:  R = 16  161 -> 54.8 s
// (R = 64 without the pairs of CTAs 0.97 ms; there a barrier of all warps per half tile took 1.50 ms,
// levels moved every tile 1.44, the MMAs issued from a loop, 200 cycles each, 1.38.)
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "dfl_pair.cuh"
#include "hzb_internal.h"
#include "kernel_math.cuh"
#include "sigma_scale.cuh"
#include "tcgen05.cuh"

namespace hzb {

static const int DX_M = 128, DX_FORM = 512, DX_THREADS = DX_FORM + 32, DX_D = 6;   // threads forming pairs, all
// largest ratio of the kernel's bounds at the smallest and the largest distance between bodies,
// up to which the common scale costs no accuracy: two spheres of 8,200 unknowns, R = 8, error here
// and of the one-directional kernel: ratio 45: 4.0e-14, 7.0e-14; 180: 5.6e-14, 7.2e-14; 363:
// 9.3e-14, 8.8e-14; 8,200: 1.3e-13, 1.0e-13
static const double DX_SPAN = 128.0;
static double dx_start(int rc) { return rc == 8 ? 0.5 : rc == 16 ? 0.8 : 1.2; }    // a CTA's start and end, in tiles
// N^2 R from which on this form is the faster one (us, here / one-directional): 900 unknowns
// (R = 16: 1.3e7) 74 / 74, 1,764 (R = 8: 2.5e7) 81 / 79, (R = 16) 85 / 117, 3,968 (R = 5) 163 / 206
static const double DX_WORK = 2.4e7;
static const int DX_RUN = 256;         // tiles after which the 64-bit sums are emptied (at most 2^54 to a tile)
static_assert((DX_RUN & (DX_RUN - 1)) == 0, "a power of two");
static const int DX_AIMG = DX_M * 64;                          // bytes of one digit image of half a tile of A
static const int DX_GEO = 3 * DFL_S * 16;                      // bytes of a tile's nodes

__host__ __device__ constexpr int dx_img(int rc) { return 2 * rc * 128; }                 // one digit image of B
__host__ __device__ constexpr int dx_stage(int rc) { return DX_D * dx_img(rc) + 2048; }    // B images and nodes
__host__ __device__ constexpr int dx_smem(int rc) { return 2 * DX_D * DX_AIMG + 2 * dx_stage(rc) + DFL_TAB * 16 + 1024; }
// tensor memory: six levels of 2 RC columns, then low and high words of the sums
__host__ __device__ constexpr int dx_cols(int rc) { return 16 * rc; }
static_assert(DX_GEO <= 2048 && dx_smem(32) <= 227 * 1024 && dx_cols(32) <= 512, "sizes");

// kind::f16 with FP16 A and B, FP32 D
__host__ __device__ constexpr uint32_t dx_idesc(int n)
{
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(DX_M >> 4) << 24);
}

// A's half tiles: K-major, 64-byte rows and swizzle (chunk c of 16 bytes of row r)
__device__ __forceinline__ uint32_t dx_chunk_off(int r, int c) { return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4)); }
// high words of the descriptors: A 512 bytes between 8-row groups, 64-byte swizzle; B as t5_desc
static const uint32_t DX_ADESC = (512u >> 4) | (1u << 14) | (4u << 29), DX_BDESC = (1024u >> 4) | (1u << 14) | (2u << 29);

// (descriptors: the low words given)
__device__ __forceinline__ void dx_mma(uint32_t d, uint32_t ad, uint32_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %6};\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}\n" ::"r"(d),
        "r"(ad), "r"(bd), "r"(idesc), "r"(acc), "r"(DX_ADESC), "r"(DX_BDESC)
        : "memory");
}

__device__ __forceinline__ void dx_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

// the same shared-memory address in the CTA of rank r of the cluster
__device__ __forceinline__ uint32_t dx_peer(uint32_t addr, uint32_t r)
{
    uint32_t d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(r));
    return d;
}
__device__ __forceinline__ void dx_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// t5_wait; CL = 2: for arrivals from both CTAs of the cluster
template <int CL>
__device__ __forceinline__ bool dx_wait(uint32_t mbar, uint32_t parity)
{
    if (CL == 1) return t5_wait(mbar, parity);
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// four columns of this warp's 32 lanes, without the wait
__device__ __forceinline__ void dx_ld4(uint32_t taddr, uint32_t (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void dx_st4(uint32_t taddr, const uint32_t (&r)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
                 "r"(r[2]), "r"(r[3])
                 : "memory");
}
__device__ __forceinline__ void dx_keep(uint32_t (&r)[4])      // uses stay behind the wait before it
{
    asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]));
}

// the six digits (integers) of x with |x| <= 2^8: five rounded to nearest, the rest in the sixth.
// The low part enters where the high part's remainder has few bits left.
__device__ __forceinline__ void dx_digits(dd x, float (&d)[DX_D])
{
    const float M = 12582912.0f;                               // 1.5 * 2^23: adding it rounds to an integer
    d[0] = (x.h + M) - M;
    float u = x.h - d[0];
    d[1] = fmaf(u, 512.f, M) - M;
    u = fmaf(u, 512.f, -d[1]);
    d[2] = fmaf(u, 512.f, M) - M;
    u = fmaf(u, 512.f, -d[2]);
    u = fmaf(x.l, 262144.f, u);
    const float c = (u + M) - M;
    d[2] += c;
    u -= c;
    d[3] = fmaf(u, 512.f, M) - M;
    u = fmaf(u, 512.f, -d[3]);
    d[4] = fmaf(u, 512.f, M) - M;
    u = fmaf(u, 512.f, -d[4]);
    d[5] = u * 512.f;
}

__device__ __forceinline__ uint32_t dx_pack(float a, float b)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
    return r;
}

template <int RC, int CL>
__global__ void __launch_bounds__(DX_THREADS, 1)
nbody_dfx_kernel(const TargetBlock *__restrict__ blocks, const int2 *__restrict__ own_tiles,
                 const int2 *__restrict__ tiles, const int *__restrict__ tile_word, int nbodies,
                 const float4 *__restrict__ ball, int ntiles, int R,
                 const float4 *__restrict__ pa, const float4 *__restrict__ pb, const float4 *__restrict__ pc,
                 const unsigned char *__restrict__ img, const int *__restrict__ key, const float4 *__restrict__ tab,
                 DflConst K, double2 *__restrict__ out, size_t split_stride, int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char dx_raw[];
    __shared__ uint32_t s_taddr;
    __shared__ __align__(8) unsigned long long s_bar[8];       // full[2]; per half tile: mma[2], formed[2]; moved, own
    __shared__ int s_rmin;
    __shared__ volatile int s_fail;
    __shared__ int s_forced;                                   // host-set flag: take the timeout exit
    __shared__ int s_exp[RC];                                  // exponents of the columns' sums
    __shared__ unsigned char s_shift[DX_FORM / 32][RC / 2];    // and of the current body's against them, by warp
    const TargetBlock tb = blocks[blockIdx.x >> 2];
    const int sub = blockIdx.x & 3;
    if (sub * DX_M >= tb.count) return;                        // whole CTA past the block's end
    constexpr int IMG = dx_img(RC), STAGE = dx_stage(RC), N = 2 * RC, CW = N / 4;   // CW: columns of a warp
    const uint32_t base = ((uint32_t)__cvta_generic_to_shared(dx_raw) + 1023u) & ~1023u;
    unsigned char *const gbase = dx_raw + (base - (uint32_t)__cvta_generic_to_shared(dx_raw));
    const uint32_t a0 = base, b0 = base + 2 * DX_D * DX_AIMG;
    unsigned char *const gb0 = gbase + 2 * DX_D * DX_AIMG;
    float4 *const s_tab = reinterpret_cast<float4 *>(gb0 + 2 * STAGE);
    const uint32_t bar0 = (uint32_t)__cvta_generic_to_shared(&s_bar[0]);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quarter = warp & 3, q4 = warp >> 2;              // rows 32 quarter + lane; sources 4 q4 .. of a half
    const int row = 32 * quarter + lane, t = sub * DX_M + row;
    for (int q = tid; q < DFL_TAB; q += DX_THREADS) s_tab[q] = tab[q];
    if (warp == 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s_taddr);
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(dx_cols(RC))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int q = 0; q < 8; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar0 + 8 * q),
                         "r"(q < 2 || q == 7 ? 1 : q < 4 ? CL : CL == 2 && q - 4 == (int)(1 - blockIdx.y % 2) ? 1 : DX_FORM / 32)
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        s_rmin = 0x7f000000;
        s_fail = 0;
        s_forced = *(volatile int *)err < 0 ? 1 : 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (CL == 2) dx_cluster_sync();                            // the barriers of both CTAs stand
    const uint32_t rank = blockIdx.y % CL, peer = rank ^ 1;
    const uint32_t tmem = s_taddr;
    // this warp's lanes and columns of level 0, and of the sums' words
    const uint32_t drow = tmem + ((uint32_t)(32 * quarter) << 16) + CW * q4;
    const uint32_t lorow = drow + DX_D * N, hirow = lorow + N;

    dd tx = {1e5f + row, 0.f}, ty = {1e5f, 0.f}, tz = {1e5f, 0.f};
    const bool live = q4 < 4 && t < tb.count;
    if (live) {
        const float4 A = pa[tb.start + t], B = pb[tb.start + t];
        tx = {A.x, B.x}; ty = {A.y, B.y}; tz = {A.z, B.z};
    }
    // the tiles of the other bodies, counted without the own body's [own.x, own.y)
    const int2 own = own_tiles[blockIdx.x >> 2];
    const int nown = own.y - own.x;
    const int i0 = (int)((long long)(ntiles - nown) * blockIdx.z / gridDim.z);
    // an injected fault ends the CTA (both of a cluster) before any copy or MMA is issued
    const int n = s_forced ? 0 : (int)((long long)(ntiles - nown) * (blockIdx.z + 1) / gridDim.z) - i0;
    auto tile_of = [&](int i) {
        const int q = i0 + i;
        return q < own.x ? q : q + nown;
    };
    // a tile whose levels start from zero: the first of a run, and every second one of a body
    auto starts = [&](int i, int word) { return (i & (DX_RUN - 1)) == 0 || !t5h_tile_odd(word); };
    auto issue = [&](int i) {
        const int tile = tile_of(i);
        const int2 tl = tiles[tile];
        const uint32_t st = b0 + (uint32_t)((i & 1) * STAGE), mb = bar0 + 8 * (i & 1), nb = (uint32_t)tl.y * 16;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(DX_D * IMG + 3 * nb)
                     : "memory");
        dx_copy(st, img + ((size_t)tile * gridDim.y + blockIdx.y) * (DX_D * IMG), DX_D * IMG, mb);
        dx_copy(st + DX_D * IMG, pa + tl.x, nb, mb);
        dx_copy(st + DX_D * IMG + DFL_S * 16, pb + tl.x, nb, mb);
        dx_copy(st + DX_D * IMG + 2 * DFL_S * 16, pc + tl.x, nb, mb);
    };
    if (tid == DX_FORM) {
        if (n > 0) issue(0);
        if (n > 1) issue(1);
    }
    int issued = min(n, 2);                                    // copies issued (the last warp's view)
    // the largest scale of the other bodies' densities (the last warp: it has no pairs to bound)
    if (q4 == 4 && lane < RC) {
        const int r = blockIdx.y * RC + lane, mine = t5h_tile_body(tile_word[own.x]);
        int k = 0;
        if (r < R)
            for (int b = 0; b < nbodies; ++b)
                if (b != mine) k = max(k, key[(size_t)b * R + r]);
        s_exp[lane] = sigma_exponent(k);
    }
    // a bound of |G| over the CTA's pairs: the distance to each tile's ball, or node by node where
    // the ball is no use (lengths of the balls: 2 pi times these)
    {
        float rm = 3e38f;
        if (live)
            for (int i = q4; i < n; i += 4) {
                const float4 b = ball[tile_of(i)];
                const float cx = 6.2831853f * tx.h - b.x, cy = 6.2831853f * ty.h - b.y, cz = 6.2831853f * tz.h - b.z;
                const float d = sqrtf(cx * cx + cy * cy + cz * cz) * 0.999f, m = d - b.w;
                if (m >= 0.5f * d) {
                    rm = fminf(rm, m * 0.15915f);
                } else {
                    const int2 tl = tiles[tile_of(i)];
                    float r2 = 3e38f;
                    for (int j = tl.x; j < tl.x + tl.y; ++j) {
                        const float4 A = pa[j], B = pb[j];
                        const float x = (tx.h - A.x) + (tx.l - B.x), y = (ty.h - A.y) + (ty.l - B.y),
                                    z = (tz.h - A.z) + (tz.l - B.z);
                        r2 = fminf(r2, x * x + y * y + z * z);
                    }
                    rm = fminf(rm, 0.999f * sqrtf(r2));
                }
            }
        for (int o = 16; o > 0; o >>= 1) rm = fminf(rm, __shfl_xor_sync(0xffffffffu, rm, o));
        if (lane == 0) atomicMin(&s_rmin, __float_as_int(rm));
    }
    const int word0 = n > 0 ? tile_word[tile_of(0)] : 0;
    // the sums start at zero
    if (q4 < 4) {
        const uint32_t z[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int q = 0; q < CW; q += 4) {
            dx_st4(lorow + q, z);
            dx_st4(hirow + q, z);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    __syncthreads();
    // 2^E: |G| <= u (u + 2 pi + |eta'|) < 2^(e + 1), u = 1 / r, e the exponent of the bound
    const float u0 = 1.0f / __int_as_float(s_rmin), bnd = 1.0001f * u0 * (u0 + K.kbound);
    const int e2 = min(max((__float_as_int(bnd) >> 23) - 127, -100), 100) + 1;
    const dd scale = {__int_as_float((127 + 8 - e2) << 23), 0.f};

    uint32_t bad = 0;                                          // columns that met a NaN
    // the shifts of a body's sums, for this warp's columns
    auto shifts = [&](int body) {
        __syncwarp();
        if (lane < CW) {
            const int c = (CW * q4 + lane) % RC, r = blockIdx.y * RC + c;
            const int e = r < R ? sigma_exponent(key[(size_t)body * R + r]) : 0;
            s_shift[warp][lane] = (unsigned char)min(max(s_exp[c] - e, 0), 62);
        }
        __syncwarp();
    };
    // the levels of the last tiles (of one body) into the sums
    auto drain = [&]() {
#pragma unroll
        for (int q = 0; q < CW; q += 4) {
            uint32_t v[DX_D][4], lo[4], hi[4];
#pragma unroll
            for (int l = 0; l < DX_D; ++l) dx_ld4(drow + l * N + q, v[l]);
            dx_ld4(lorow + q, lo);
            dx_ld4(hirow + q, hi);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int l = 0; l < DX_D; ++l) dx_keep(v[l]);
            dx_keep(lo);
            dx_keep(hi);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                // units of 2^-32: levels 3, 4, 5 rounded together
                const float low = fmaf(__uint_as_float(v[5][c]), 0x1p-13f,
                                       fmaf(__uint_as_float(v[4][c]), 0x1p-4f, 32.f * __uint_as_float(v[3][c])));
                if (low != low) bad |= 1u << (q + c);
                long long s = (long long)__float2int_rn(low);
                s += (long long)__float2int_rn(__uint_as_float(v[2][c])) * (1 << 14);
                s += (long long)__float2int_rn(__uint_as_float(v[1][c])) * (1 << 23);
                s += (long long)((unsigned long long)(unsigned)__float2int_rn(__uint_as_float(v[0][c])) << 32);
                const int d = s_shift[warp][q + c];
                s = (s + ((1ll << d) >> 1)) >> d;
                s += (long long)(((unsigned long long)hi[c] << 32) | lo[c]);
                lo[c] = (uint32_t)s;
                hi[c] = (uint32_t)((unsigned long long)s >> 32);
            }
            dx_st4(lorow + q, lo);
            dx_st4(hirow + q, hi);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    };
    // the sums into the output, which holds what earlier ones left (begun); then they start at zero
    bool begun = false, failed = false;
    auto emit = [&]() {
        const double f = 0x1p-40 / (double)scale.h;            // 2^-32 of the unit, 2^-8 of the densities
#pragma unroll 1
        for (int q = 0; q < CW; q += 4) {
            uint32_t lo[4], hi[4];
            const uint32_t z[4] = {0u, 0u, 0u, 0u};
            __syncwarp();
            dx_ld4(lorow + q, lo);
            dx_ld4(hirow + q, hi);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            dx_keep(lo);
            dx_keep(hi);
            dx_st4(lorow + q, z);
            dx_st4(hirow + q, z);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                // columns CW q4 ..: the first RC are real parts, the others imaginary parts
                const int col = CW * q4 + q + c, r = blockIdx.y * RC + col % RC;
                if (!live || r >= R) continue;
                const long long s = (long long)(((unsigned long long)hi[c] << 32) | lo[c]);
                double v = (double)s * f * sigma_pow2(s_exp[col % RC]);
                double *o = reinterpret_cast<double *>(out + blockIdx.z * split_stride + (size_t)(tb.start + t) * R + r) + col / RC;
                if (begun) v += *o;
                *o = (failed || (bad >> (q + c) & 1)) ? __longlong_as_double(0x7ff8000000000000ll) : v;
            }
        }
        __syncwarp();
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        begun = true;
    };
    bool ok = s_forced == 0;
    if (q4 == 4) {
        // the last warp: MMAs of each half tile once all 16 have formed it, copies into free stages;
        // every wait gives one answer to all lanes
        int halves = 0, armed = 0, moves = 0;                  // half tiles' MMAs issued, other halves announced, drains
        auto wait = [&](uint32_t mbar, int phase) { return t5_all(dx_wait<CL>(mbar, (uint32_t)(phase & 1))); };
        auto arm = [&]() {                                     // the other half of a tile comes from the other CTA
            if (lane == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar0 + 32 + 8 * peer),
                             "r"(DX_D * DX_AIMG)
                             : "memory");
            ++armed;
        };
        int next = word0;
        for (int i = 0; i < n && ok; ++i) {
            const bool first = starts(i, next);
            if (i + 1 < n) next = tile_word[tile_of(i + 1)];
            if (i > 0) {
                ok = (CL == 1 || wait(bar0 + 16, i - 1)) && wait(bar0 + 24, i - 1);
                if (ok && i + 1 < n) {
                    if (lane == 0) issue(i + 1);
                    issued = i + 2;
                }
            }
            if (CL == 2) arm();
            // (CL = 1: the warps that form the halves have waited for the images)
            if (CL == 2) ok = ok && wait(bar0 + 8 * (i & 1), i >> 1);
#pragma unroll 1
            for (int hh = 0; hh < 2 && ok; ++hh) {
                const int h = CL == 2 ? (int)rank ^ hh : hh;   // CL = 2: the own half first
                ok = wait(bar0 + 32 + 8 * h, i) && !__any_sync(0xffffffffu, s_fail);
                if (CL == 2 && ok && hh == 0 && lane == 0)
                    asm volatile(
                        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            dx_peer(a0 + rank * (DX_D * DX_AIMG), peer)),
                        "r"(a0 + rank * (DX_D * DX_AIMG)), "r"(DX_D * DX_AIMG), "r"(dx_peer(bar0 + 32 + 8 * rank, peer))
                        : "memory");
                // (CL = 1: the warps that formed the half have moved the levels)
                if (CL == 2 && ok && hh == 0 && i > 0 && first) ok = wait(bar0 + 48, moves++);
                if (!ok) break;
                __syncwarp();
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (t5_elect()) {
                    // (unrolled: in a loop the address arithmetic of one MMA took this warp 200 cycles)
                    const uint32_t ad = ((a0 + h * (DX_D * DX_AIMG)) & 0x3FFFF) >> 4 | (1u << 16);
                    const uint32_t bd = (uint32_t)t5_desc(b0 + (uint32_t)((i & 1) * STAGE) + 64 * h);
                    const uint32_t more = first ? hh : 1;
#pragma unroll
                    for (int l = 0; l < DX_D; ++l)
#pragma unroll
                        for (int a = 0; a <= l; ++a)
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks)
                                dx_mma(tmem + l * N, ad + ((a * DX_AIMG + 32 * ks) >> 4), bd + (((l - a) * IMG + 32 * ks) >> 4),
                                       dx_idesc(N), a | ks ? 1u : more);
                    if (CL == 1)
                        asm volatile(
                            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar0 + 16 + 8 * h)
                            : "memory");
                    else
                        asm volatile(
                            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
                            "[%0], %1;" ::"r"(bar0 + 16 + 8 * h), "h"((unsigned short)3)
                            : "memory");
                }
                __syncwarp();
                ++halves;
            }
        }
        if (!ok) s_fail = 1;
        // what is in flight (after a timeout: once more, the other CTA's half among it, which that CTA
        // may have sent before its own wait ran out)
        if (CL == 2 && !ok && armed > 0) dx_wait<CL>(bar0 + 32 + 8 * peer, (uint32_t)((armed - 1) & 1));
        __syncwarp();
        if (halves > 0) {
            if (t5_elect())
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar0 + 56)
                             : "memory");
            __syncwarp();
            ok &= t5_wait(bar0 + 56, 0u);
        }
        for (int i = max(0, issued - 2); i < issued; ++i) ok &= t5_wait(bar0 + 8 * (i & 1), (uint32_t)((i >> 1) & 1));
    } else {
        int next = word0, body = t5h_tile_body(word0);         // body: of the levels
        if (n > 0) shifts(body);
        auto moved = [&]() {                                   // the levels are free for the next MMAs
            if (CL == 1) return;                               // (known from the half that this warp forms next)
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar0 + 48) : "memory");
        };
        // runs of the tiles that the sums hold
        for (int run0 = 0; run0 < n && ok; run0 += DX_RUN) {
            const int run1 = min(n, run0 + DX_RUN);
            for (int i = run0; i < run1; ++i) {
                const int word = next, cnt = t5h_tile_count(word);
                const bool first = starts(i, word);
                if (i + 1 < n) next = tile_word[tile_of(i + 1)];
                ok = t5_wait(bar0 + 8 * (i & 1), (uint32_t)((i >> 1) & 1));
                const float4 *const S = reinterpret_cast<const float4 *>(gb0 + (i & 1) * STAGE + DX_D * IMG);
#pragma unroll 1
                for (int h = CL == 2 ? (int)rank : 0; h < (CL == 2 ? (int)rank + 1 : 2); ++h) {
                    uint32_t dig[DX_D][4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const int j = 16 * h + 4 * q4 + v;
                        if (j < cnt) {
                            const float4 A4 = S[j], B4 = S[DFL_S + j], C4 = S[2 * DFL_S + j];
                            const DflGeom G = dfl_geom<2>(tx, ty, tz, A4, B4, scale, s_tab, K);
                            dd gr, gi;
                            dfl_kernel_value(G, dfl_projection({A4.w, B4.w}, {C4.x, C4.z}, {C4.y, C4.w}, G), K, gr, gi);
                            float dr[DX_D], di[DX_D];
                            dx_digits(gr, dr);
                            dx_digits(gi, di);
#pragma unroll
                            for (int l = 0; l < DX_D; ++l) dig[l][v] = dx_pack(dr[l], di[l]);
                        } else {
#pragma unroll
                            for (int l = 0; l < DX_D; ++l) dig[l][v] = 0u;
                        }
                    }
                    if (i > 0) ok &= dx_wait<CL>(bar0 + 16 + 8 * h, (uint32_t)((i - 1) & 1));   // A's half is free
                    // (CL = 2: both halves every tile, so that no phase of a barrier goes by unseen)
                    if (i > 0 && (CL == 2 || (h == 0 && first)))
                        ok &= dx_wait<CL>(bar0 + 16 + 8 * (h ^ 1), (uint32_t)((i - 1) & 1));
                    if ((CL == 2 || h == 0) && i > run0 && first) {   // the tiles since the last start are through: their levels
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        __syncwarp();
                        drain();
                        moved();
                    }
                    if (body != t5h_tile_body(word)) shifts(body = t5h_tile_body(word));
                    const uint32_t at = a0 + h * (DX_D * DX_AIMG) + dx_chunk_off(row, q4);
#pragma unroll
                    for (int l = 0; l < DX_D; ++l) t5_st4(at + l * DX_AIMG, dig[l][0], dig[l][1], dig[l][2], dig[l][3]);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    if (__any_sync(0xffffffffu, !ok)) s_fail = 1;  // ends the MMAs, and below the loop
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar0 + 32 + 8 * h) : "memory");
                }
                if (__any_sync(0xffffffffu, s_fail)) {
                    ok = false;
                    break;
                }
            }
            if (ok) {                                              // the run's last tiles
                ok = t5_all(dx_wait<CL>(bar0 + 16, (uint32_t)((run1 - 1) & 1))) &&
                     t5_all(dx_wait<CL>(bar0 + 24, (uint32_t)((run1 - 1) & 1)));
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                drain();
                if (run1 < n) {
                    emit();
                    moved();
                }
            }
        }
        if (__any_sync(0xffffffffu, !ok)) s_fail = 1;
    }
    failed = __syncthreads_or(!ok);
    if (q4 < 4) emit();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(dx_cols(RC)) : "memory");
    if (CL == 2) dx_cluster_sync();                            // no stores or arrivals into a CTA that has ended
    if (failed && tid == 0 && !s_forced) atomicExch(err, 1);   // (a negative flag stays for all CTAs of the launch)
}

// key[b R + r]: the largest high word of |Re|, |Im| of w_j sigma_{j,r} c0 over the finite values of
// body b (rounded up; 0: none), so that these are below 2^sigma_exponent(key).  A warp takes eight
// columns of a tile, a lane one of them and eight sources.
__global__ void dfx_key_kernel(int ntiles, int R, int per, const int2 *__restrict__ tiles, const int *__restrict__ tile_word,
                               const double4 *__restrict__ pos, const double2 *__restrict__ sigma, double c0,
                               int *__restrict__ key)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)ntiles * per * 32) return;
    const int lane = threadIdx.x & 31, tile = (int)(e / 32 / per), col = (int)(e / 32 % per) * 8 + (lane & 7);
    const int2 tl = tiles[tile];
    int big = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int s = 8 * (lane >> 3) + q;
        if (s < tl.y && col < R) {
            const double2 v = sigma[(size_t)(tl.x + s) * R + col];
            const double wq = pos[tl.x + s].w * c0;
            const int hx = __double2hiint(v.x * wq) & 0x7fffffff, hy = __double2hiint(v.y * wq) & 0x7fffffff;
            big = max(big, max(hx < 0x7ff00000 ? hx : 0, hy < 0x7ff00000 ? hy : 0));
        }
    }
    big = max(big, __shfl_xor_sync(0xffffffffu, big, 8));
    big = max(big, __shfl_xor_sync(0xffffffffu, big, 16));
    if (lane < 8 && col < R && big) atomicMax(&key[(size_t)t5h_tile_body(tile_word[tile]) * R + col], big + 1);
}

// Digit images of s = 2^8 w sigma c0, scaled below 2^8 per body and column (key): for every tile and chunk of
// RC right-hand sides DX_D images of 2 RC rows of 128 bytes, the values of the 32 sources along a
// row: column r (real part of y) holds (Re s, -Im s) per source, column RC + r (Im s, Re s).
// One thread per (tile, column, four sources).
__global__ void dfx_density_kernel(int ntiles, int R, int rc, int nchunk, const int2 *__restrict__ tiles,
                                   const int *__restrict__ tile_word, const double4 *__restrict__ pos,
                                   const double2 *__restrict__ sigma, double c0, const int *__restrict__ key, unsigned char *__restrict__ img)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int ncol = rc * nchunk;
    if (e >= (size_t)ntiles * ncol * 8) return;
    const int col = (int)(e % ncol), g = (int)(e / ncol % 8), tile = (int)(e / ncol / 8);
    const int2 tl = tiles[tile];
    const double sc = col < R ? c0 * sigma_pow2(8 - sigma_exponent(key[(size_t)t5h_tile_body(tile_word[tile]) * R + col])) : 0.0;
    uint32_t re[DX_D][4], im[DX_D][4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int s = 4 * g + v;
        dd x = {0.f, 0.f}, y = {0.f, 0.f};
        if (s < tl.y && col < R) {
            const double wq = pos[tl.x + s].w * sc;
            const double2 z = sigma[(size_t)(tl.x + s) * R + col];
            x = split(z.x * wq);
            y = split(z.y * wq);
        }
        float dr[DX_D], di[DX_D];
        dx_digits(x, dr);
        dx_digits(y, di);
#pragma unroll
        for (int l = 0; l < DX_D; ++l) {
            re[l][v] = dx_pack(dr[l], -di[l]);
            im[l][v] = dx_pack(di[l], dr[l]);
        }
    }
    const int n = col % rc;
    unsigned char *b = img + ((size_t)tile * nchunk + col / rc) * (DX_D * dx_img(rc));
#pragma unroll
    for (int l = 0; l < DX_D; ++l, b += dx_img(rc)) {
        *reinterpret_cast<uint4 *>(b + t5_chunk_off(n, g)) = make_uint4(re[l][0], re[l][1], re[l][2], re[l][3]);
        *reinterpret_cast<uint4 *>(b + t5_chunk_off(n + rc, g)) = make_uint4(im[l][0], im[l][1], im[l][2], im[l][3]);
    }
}

// ---------------------------------------------------------------- host

// Whether the sum of R right-hand sides takes this form (an error: *st).
bool dfx_usable(hzb_ctx *c, int R, hzb_status *st)
{
    *st = HZB_OK;
    if (R < 3 || (double)c->N * c->N * R < DX_WORK) return false;
    if ((*st = ensure_t5h(c))) return false;
    return c->t5h_span > 0.0 && c->t5h_span < DX_SPAN;
}

hzb_status interbody_dfx(hzb_ctx *c, int R, const double2 *sigma, double2 *y)
{
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->opt.device);
    const int rc = R <= 8 ? 8 : R <= 16 ? 16 : 32, nt = c->t5h_ntiles, most = c->t5h_most;
    const int cl = R > 32 ? 2 : 1, nchunk = ((R + rc - 1) / rc + cl - 1) / cl * cl;
    hzb_status st = ensure_dfl(c);
    if (st) return st;
    // Source chunks: the shortest time, in tiles.  Bodies of one size: whole waves of equal CTAs;
    // others: the mean load and most of a long CTA's time at the end.  A partial sum costs 1e-6 of a
    // tile.  Beyond 32 waves there is nothing left to fill, and the partial sums stay below 0.4 GB
    // (128 x 32 values to a CTA).
    const long long ctas = (long long)c->t5h_ctas * nchunk;
    const bool even = c->t5h_mean > 0.97 * most;
    int nsplit = 1;
    double best = 1e300;
    for (int ns = 1; ns <= std::min(64, most) && (ns == 1 || ns * ctas <= 32LL * sms); ++ns) {
        const double one = std::ceil((double)most / ns) + dx_start(rc);
        const double tt = (even ? std::ceil((double)(ns * ctas) / sms) * one
                                : std::max(one, ctas * (c->t5h_mean + ns * dx_start(rc)) / sms + 0.6 * one)) +
                          1e-6 * (double)c->N * R * ns;
        if (tt < best) { best = tt; nsplit = ns; }
    }
    const size_t n = (size_t)c->N * R;
    double2 *out = y;
    if (nsplit > 1) {
        if (check_cuda(c, c->nb_part64.ensure(n * nsplit), "alloc partial sums")) return HZB_ENOMEM;
        out = c->nb_part64.ptr;
    }
    if (check_cuda(c, c->t5h_img.ensure((size_t)nt * nchunk * DX_D * dx_img(rc)), "alloc operand images") ||
        check_cuda(c, c->dlkey.ensure((size_t)c->t5h_nbodies * R), "alloc scales"))
        return HZB_ENOMEM;
    if ((st = tc_flag_begin(c, FAULT_TIMEOUT))) return st;
    const double s = c->k / (2.0 * M_PI), c0 = s * s / (4.0 * M_PI);
    c->interbody_calls++;
    const int slot = prof_begin(c, 2);
    if (check_cuda(c, cudaMemsetAsync(c->dlkey.ptr, 0, (size_t)c->t5h_nbodies * R * sizeof(int), c->stream), "clear scales"))
        return HZB_ECUDA;
    const int per = (R + 7) / 8;
    const size_t nk = (size_t)nt * per * 32, ne = (size_t)nt * rc * nchunk * 8;
    dfx_key_kernel<<<(unsigned)((nk + 255) / 256), 256, 0, c->stream>>>(nt, R, per, c->t5h_tiles.ptr, c->t5h_words,
                                                                      c->pos64.ptr, sigma, c0, c->dlkey.ptr);
    dfx_density_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, c->stream>>>(nt, R, rc, nchunk, c->t5h_tiles.ptr,
                                                                          c->t5h_words, c->pos64.ptr, sigma, c0,
                                                                          c->dlkey.ptr, c->t5h_img.ptr);
    const dim3 grid((unsigned)c->n_tblocks * 4, nchunk, nsplit);
    const float4 *ball = reinterpret_cast<const float4 *>(c->t5h_src.ptr + (size_t)nt * 6 * DFL_S);
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kern) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dx_smem(rc));
        if (e != cudaSuccess) return;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(DX_THREADS);
        cfg.dynamicSmemBytes = dx_smem(rc);
        cfg.stream = c->stream;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1;
        at[0].val.clusterDim.y = cl;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = cl > 1 ? 1 : 0;
        e = cudaLaunchKernelEx(&cfg, kern, (const TargetBlock *)c->tblocks.ptr, (const int2 *)(c->t5h_tiles.ptr + nt),
                               (const int2 *)c->t5h_tiles.ptr, c->t5h_words, c->t5h_nbodies, ball, nt, R,
                               (const float4 *)c->dla.ptr,
                               (const float4 *)c->dlb.ptr, (const float4 *)c->dlc.ptr,
                               (const unsigned char *)c->t5h_img.ptr, (const int *)c->dlkey.ptr,
                               (const float4 *)c->dfltab.ptr, dfl_constants(c), out, n, c->kerr.ptr);
        if (e != cudaSuccess) return;
        e = cudaGetLastError();
    };
    if (rc == 8) launch(nbody_dfx_kernel<8, 1>);
    else if (rc == 16) launch(nbody_dfx_kernel<16, 1>);
    else if (cl == 1) launch(nbody_dfx_kernel<32, 1>);
    else launch(nbody_dfx_kernel<32, 2>);
    c->launches += 3;
    if (check_cuda(c, e, "nbody_dfx_kernel")) return HZB_ECUDA;
    if (nsplit > 1) {
        if ((st = dfl_split_reduce(c, n, nsplit, out, y))) return st;
        c->launches++;
    }
    prof_end(c, slot);
    return tc_flag_end(c, "nbody_dfx_kernel", false);      // queued, as the other double-float sums are
}

}  // namespace hzb
