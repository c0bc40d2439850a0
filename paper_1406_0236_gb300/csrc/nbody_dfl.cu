// Inter-body sum y = B sigma (Sec. 3.3, Eq. (nystromnaive)) in lean double-float
// arithmetic on the FP32 pipe: the refinement residual's sum of the mixed-precision
// solve at about the accuracy of FP64 (measured max-norm error against the oracle
// ~1e-13 of max |y|), without the FP64 pipe (1/64 of the FP32 rate on GB300).
//
// Up to two right-hand sides each unordered pair of nodes on different bodies is evaluated
// once for both directions (the block-pair scheme of nbody_sym.cu: 32-source tiles met in 32
// rotation steps, source-side sums moving one lane per step, FP64 atomic adds into y);
// above, a one-directional kernel shares the pair's work among up to 32 right-hand sides (where
// the tensor-core sums of nbody_dfx.cu do not apply: short sums, nearly touching bodies, k = 0).
//
// Lengths are in wavelengths (x k / 2 pi, split into hi + lo after scaling; unscaled when
// k = 0), so that r is the phase in turns and no rounding stands between them.  With
// d = x_i - x_j, r = |d|, E = e^{2 pi i r} / r, kr = 2 pi r, eta' = 2 pi eta / k:
//     w_j K(x_i, x_j) = (k / 2 pi)^2 w_j / (4 pi) E [X_1 - i (kr X_1 + eta')],  X_1 =  n_j.d / r^2,
//     w_i K(x_j, x_i) = (k / 2 pi)^2 w_i / (4 pi) E [X_2 - i (kr X_2 + eta')],  X_2 = -n_i.d / r^2;
// E, r and kr are shared by the two directions.  The densities come weighted, scaled per
// right-hand side by a power of two to |sigma'| < 1 (y is scaled back), and split once per
// call (dfl_sigma_*_kernel).
//
// Arithmetic: lean double-float (lean_df.cuh): error-free products and sums left
// unnormalised.  Sums whose magnitude is bounded beforehand are taken on a fixed grid instead
// of by two-sums: adding a product to m = 1.5 * 2^E rounds it to a multiple of ulp(m) in the
// product's own fused multiply-add (s = a b + m), s - m is exact, and so is what is left,
// fma(a, b, -(s - m)): three operations where a product and a two-sum take eight.  So are
//   * n.d (bounded by r), kr X + eta' (by 2 pi + |eta'|) and the angle addition (by 1, with
//     the table on the grid of ulp(3));
//   * the sums over sources of the one-directional kernel for five and more right-hand sides
//     (DflGrid): the mantissas of s enter an integer sum (exact), the remainders an FP32 sum
//     whose whole units are carried over every four sources, and both a running double-float
//     sum once per tile of 32.  28 issue slots per complex multiply-add instead of 48.  The
//     remainders have FP32's 24 bits below a grid 22 bits below the largest product, so that
//     the grid has to be tight: it follows the magnitude of each pair's kernel (weight
//     included), and the densities are scaled up to one tile by tile.  A short sum (below
//     DFL_GRID_MIN sources) keeps two-sums: their error grows with the running sum.
// 1/r: the hardware estimate of 1/sqrt(r^2) and one Halley step (cubic convergence, so the
// estimate's 2^-23 error falls below 2^-60); r: r^2 / r rounded, and its residual.
// e^{2 pi i r}: r is reduced to [-1/2, 1/2] turns and then to the nearest of 1024 table
// angles (shared memory); the remainder |delta| <= pi / 1024 enters through
// cos(delta) - 1 = -delta^2/2 + delta^4/24 and sin(delta) = delta - delta^3/6 + delta^5/120
// (truncation below 1e-17) and angle addition.
// The translation unit is compiled with -fmad=false so that the compiler never fuses
// the separately rounded operations these transformations depend on.
//
// Both kernels are bound by the issue of FP32 instructions (78 % of the issue slots used, the
// rest lost to register-port conflicts): about 200 for a pair's geometry and phase, 100 more
// and the sums' 96 for the second direction.  One pass of the earlier form (two-sums
// throughout, lengths unscaled) and of this one, and the error of each against 64 bits:
//   29,280 unknowns, k = 6:  R = 1  4.49 -> 4.10 ms, 1.8e-13 -> 1.1e-13;  R = 8  15.5 -> 11.0;
//                            R = 16  25.6 -> 16.6;  R = 64  98.6 -> 61.0 ms, 2.8e-13 -> 1.2e-13
//   8,200 unknowns, k = 2:   R = 4  0.68 -> 0.51 ms, 6.0e-14 -> 5.0e-14;
//                            R = 64  5.62 -> 3.73 ms, 7.6e-14 -> 5.7e-14
#include <algorithm>
#include <cmath>
#include <vector>

#include "dfl_pair.cuh"
#include "hzb_internal.h"
#include "lean_df.cuh"
#include "sigma_scale.cuh"

namespace hzb {

using namespace lean;

static const int DFL_T = 512;          // targets of a TargetBlock
static const int DFL_NT = 256;         // threads (targets) per CTA of the one-directional kernel
// sources of a target from which on the sums run on a grid: at 4,100 sources the grid's error
// is that of the two-sums it replaces (5.7e-14 against 6e-14), at 216 it would be twice it
static const int DFL_GRID_MIN = 4096;

// A sum over a tile: integers in units of the tile's finest grid (modulo 2^32: the mantissas of m in
// them pass that many times), and the remainders.
struct DflAcc {
    unsigned v;
    float l;
};

// The grids of a tile: a pair of kernel magnitude |G| rounds its products to the multiples of
// ulp(m), m = dfl_magic_of(max(|Re G|, |Im G|)) (|sigma'| < 1 / sqrt 2, so |G sigma'| stays in
// m's binade), but to none finer than `fine`, three binades below the tile's bound of |G|;
// its mantissas enter the integer sums times mult = ulp(m) / ulp(fine).
struct DflGrid {
    float m;
    unsigned mult;
};

__device__ __forceinline__ float dfl_fine(float rmin, float kbound, float wmax)
{
    const float u = 1.0f / rmin;                           // |G| <= w (1/r) (1/r + 2 pi + |eta'|)
    return __int_as_float(__float_as_int(dfl_magic_of(1.0001f * wmax * u * (u + kbound))) - (3 << 23));
}

__device__ __forceinline__ DflGrid dfl_grid(float g, float fine)
{
    const int fb = __float_as_int(fine);
    const int mb = max((__float_as_int(g) & 0x7f800000) + 0x01400000, fb);
    return {__int_as_float(mb), 1u << ((mb - fb) >> 23)};
}

// acc += a b + c d on the grid of one pair.  v collects the mantissas of s with those of m in
// them: the caller subtracts the sum of m's mantissas once for all accumulators (dfl_flush).
__device__ __forceinline__ void dfl_mac2(DflAcc &acc, dd a, dd b, dd c, dd d, DflGrid g)
{
    const float s1 = fmaf(a.h, b.h, g.m), t1 = s1 - g.m, l1 = fmaf(a.h, b.h, -t1);
    const float s2 = fmaf(c.h, d.h, s1), t2 = s2 - s1, l2 = fmaf(c.h, d.h, -t2);
    float x = a.h * b.l;
    x = fmaf(a.l, b.h, x);
    x = fmaf(c.h, d.l, x);
    x = fmaf(c.l, d.h, x);
    acc.v = __float_as_uint(s2) * g.mult + acc.v;
    acc.l += (l1 + l2) + x;
}

// whole units of the remainders into the integers (|l| stays about one unit)
__device__ __forceinline__ void dfl_carry(DflAcc &acc, float fine)
{
    const float s = acc.l + fine;
    acc.v += __float_as_uint(s) - __float_as_uint(fine);
    acc.l -= s - fine;
}

// run += sc acc, the tile's sum (v - corr below 2^31, sc a power of two), normalised; acc = 0
__device__ __forceinline__ dd dfl_flush(dd run, DflAcc &acc, unsigned corr, float ulp, float sc)
{
    const float us = ulp * sc;
    const int v = (int)(acc.v - corr);
    const dd a = two_sum(run.h, __int2float_rn(v & ~255) * us);
    const dd b = two_sum(a.h, __int2float_rn(v & 255) * us);
    const dd r = norm({b.h, run.l + fmaf(acc.l, sc, a.l + b.l)});
    acc = {0u, 0.f};
    return r;
}

// the power of two that brings values up to the one with these bits below one (and back)
__device__ __forceinline__ float dfl_up(int bits)
{
    const int e = bits >> 23;                              // 0: all zero; 255: not finite
    return (e < 1 || e > 252) ? 1.0f : __int_as_float((253 - e) << 23);
}
__device__ __forceinline__ float dfl_down(int bits)
{
    const int e = bits >> 23;
    return (e < 1 || e > 252) ? 1.0f : __int_as_float((e + 1) << 23);
}
__device__ __forceinline__ int dfl_bits(float4 v)          // of sqrt 2 times the modulus, rounded up
{
    return __float_as_int(1.4144f * sqrtf(v.x * v.x + v.z * v.z));
}
__device__ __forceinline__ float4 dfl_times(float4 v, float s)
{
    return make_float4(v.x * s, v.y * s, v.z * s, v.w * s);
}

// A ball about a tile's sources (x, y, z, radius), by one warp whose lanes hold them.
__device__ __forceinline__ float4 dfl_ball(float4 a, bool have, int cnt)
{
    float x = have ? a.x : 0.f, y = have ? a.y : 0.f, z = have ? a.z : 0.f;
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    const float ic = 1.0f / cnt;
    x *= ic; y *= ic; z *= ic;
    const float dx = a.x - x, dy = a.y - y, dz = a.z - z;
    float r = have ? sqrtf(dx * dx + dy * dy + dz * dz) : 0.f;
    for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
    // rounding of the centre, the radius and the distances measured from it
    return make_float4(x, y, z, r * 1.0001f + 1e-6f * (fabsf(x) + fabsf(y) + fabsf(z)));
}

// Lower bound of the distance from a target to a tile's sources: through the ball, or, where
// the ball is no use (closer than its own size), over the sources.
__device__ __forceinline__ float dfl_rmin(dd tx, dd ty, dd tz, float4 ball, const float4 *a, const float4 *b, int cnt)
{
    const float dx = tx.h - ball.x, dy = ty.h - ball.y, dz = tz.h - ball.z;
    const float dist = sqrtf(dx * dx + dy * dy + dz * dz) * 0.9999f - 1e-6f * (fabsf(tx.h) + fabsf(ty.h) + fabsf(tz.h));
    float rm = dist - ball.w;
    if (rm < 0.5f * dist) {
        float r2 = 3.0e38f;
        for (int j = 0; j < cnt; ++j) {
            const float x = (tx.h - a[j].x) + (tx.l - b[j].x), y = (ty.h - a[j].y) + (ty.l - b[j].y),
                        z = (tz.h - a[j].z) + (tz.l - b[j].z);
            r2 = fminf(r2, x * x + y * y + z * z);
        }
        rm = 0.999f * sqrtf(r2);
    }
    return rm;
}

// ---------------------------------------------------------------- densities

static const int DFL_SIG_SMALL = 2048;    // N x R up to which one block does both passes

// key[r] = largest high word of |Re|, |Im| of w_j sigma_{j,r} c0 over the finite ones
__device__ __forceinline__ int dfl_key(double2 v, double w, double c0)
{
    const int hx = __double2hiint(v.x) & 0x7fffffff, hy = __double2hiint(v.y) & 0x7fffffff;
    const int h = __double2hiint(__hiloint2double(max(hx, hy) | 1, 0) * (w * c0));
    return h < 0x7ff00000 ? h + 1 : 0;                     // + 1: the low words dropped above
}

__device__ __forceinline__ float4 dfl_sigma(double2 v, double w, double c0, int key)
{
    const double sc = sigma_pow2(-sigma_exponent(key)), wq = w * c0;
    return csplit(make_double2(v.x * wq * sc, v.y * wq * sc));
}

// grid (blocks, ceil(R / 256)): 256 threads over up to 256 right-hand sides
__global__ void __launch_bounds__(256)
dfl_sigma_max_kernel(long long N, int R, const double4 *__restrict__ pos, const double2 *__restrict__ sigma, double c0,
                     int weighted, int *__restrict__ key)
{
    __shared__ int s_key[256];
    const int cols = min(R - (int)blockIdx.y * 256, 256), rows = 256 / cols;
    const int c = threadIdx.x % cols, row = threadIdx.x / cols, r = blockIdx.y * 256 + c;
    s_key[threadIdx.x] = 0;
    __syncthreads();
    int m = 0;
    if (row < rows)
        for (long long i = (long long)blockIdx.x * rows + row; i < N; i += (long long)gridDim.x * rows)
            m = max(m, dfl_key(sigma[i * R + r], weighted ? pos[i].w : 1.0, c0));
    if (m) atomicMax(&s_key[c], m);
    __syncthreads();
    if ((int)threadIdx.x < cols && s_key[threadIdx.x]) atomicMax(&key[blockIdx.y * 256 + threadIdx.x], s_key[threadIdx.x]);
}

__global__ void dfl_sigma_split_kernel(size_t n, int R, const double4 *__restrict__ pos,
                                       const double2 *__restrict__ sigma, double c0, int weighted,
                                       const int *__restrict__ key, float4 *__restrict__ out)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) out[e] = dfl_sigma(sigma[e], weighted ? pos[e / R].w : 1.0, c0, key[e % R]);
}

// both passes in one block (R <= 64)
__global__ void __launch_bounds__(1024)
dfl_sigma_small_kernel(int n, int R, const double4 *__restrict__ pos, const double2 *__restrict__ sigma, double c0,
                       int weighted, int *__restrict__ key, float4 *__restrict__ out)
{
    __shared__ int s_key[64];
    if (threadIdx.x < 64) s_key[threadIdx.x] = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < n; e += 1024) 
        atomicMax(&s_key[e % R], dfl_key(sigma[e], weighted ? pos[e / R].w : 1.0, c0));
    __syncthreads();
    if ((int)threadIdx.x < R) key[threadIdx.x] = s_key[threadIdx.x];
    for (int e = threadIdx.x; e < n; e += 1024)
        out[e] = dfl_sigma(sigma[e], weighted ? pos[e / R].w : 1.0, c0, s_key[e % R]);
}

__global__ void dfl_nodes_kernel(long long N, const double4 *__restrict__ pos, const double4 *__restrict__ nrm,
                                 double3 o, double s, float4 *__restrict__ a, float4 *__restrict__ b,
                                 float4 *__restrict__ cn, float2 *__restrict__ w)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double4 p = pos[i], n = nrm[i];
    const dd x = split((p.x - o.x) * s), y = split((p.y - o.y) * s), z = split((p.z - o.z) * s);
    const dd nx = split(n.x), ny = split(n.y), nz = split(n.z);
    a[i] = make_float4(x.h, y.h, z.h, nx.h);
    b[i] = make_float4(x.l, y.l, z.l, nx.l);
    cn[i] = make_float4(ny.h, nz.h, ny.l, nz.l);
    const dd wd = split(p.w);
    w[i] = make_float2(wd.h, wd.l);
}

// ---------------------------------------------------------------- pair-symmetric kernel

// Source j of a tile, staged in shared memory: position and normal (hi, lo split as
// in the node arrays) and sigma'_j for RC right-hand sides.
template <int RC>
struct DflTile {
    float4 a[DFL_S], b[DFL_S], c[DFL_S];
    float4 sig[DFL_S][RC];                                // re.hi, re.lo, im.hi, im.lo of sigma'
};

template <int RC>
__global__ void __launch_bounds__(DFL_T, 1)
nbody_dfl_sym_kernel(const int2 *__restrict__ pairs, const TargetBlock *__restrict__ blocks, int R,
                     const float4 *__restrict__ pa, const float4 *__restrict__ pb, const float4 *__restrict__ pc,
                     const float4 *__restrict__ sdd, const int *__restrict__ key, const float4 *__restrict__ tab,
                     DflConst K, double2 *__restrict__ y, SymSplit sp)
{
    __shared__ DflTile<RC> s_tile[2];                     // double-buffered source tiles
    __shared__ float4 s_tab[DFL_TAB];
    const int2 pr = pairs[blockIdx.x];
    const TargetBlock bi = blocks[pr.x], bj = blocks[pr.y];
    // this CTA's sources [jlo, jhi) of J and rotation steps [st0, st1) of each tile
    const int jlo = (blockIdx.z / sp.nstep) * sp.jchunk, jhi = min(bj.count, jlo + sp.jchunk);
    const int st0 = (blockIdx.z % sp.nstep) * (DFL_S / sp.nstep), st1 = st0 + DFL_S / sp.nstep;
    if (jlo >= jhi) return;
    const int r0 = blockIdx.y * RC;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int q = tid; q < DFL_TAB; q += DFL_T) s_tab[q] = tab[q];
    const bool live = tid < bi.count;
    dd tx = {1e5f + tid, 0.f}, ty = {1e5f, 0.f}, tz = {1e5f, 0.f};
    dd mx = {0.f, 0.f}, my = {0.f, 0.f}, mz = {0.f, 0.f};
    dd wr[RC], wi[RC], atr[RC], ati[RC];
    double scale[RC];
#pragma unroll
    for (int c = 0; c < RC; ++c) {
        wr[c] = wi[c] = atr[c] = ati[c] = {0.f, 0.f};
        scale[c] = r0 + c < R ? sigma_pow2(sigma_exponent(key[r0 + c])) : 0.0;
    }
    if (live) {
        const int g = bi.start + tid;
        const float4 A = pa[g], B = pb[g], C = pc[g];
        tx = {A.x, B.x}; ty = {A.y, B.y}; tz = {A.z, B.z};
        mx = {-A.w, -B.w}; my = {-C.x, -C.z}; mz = {-C.y, -C.w};      // negated: X_2 = -n_i.d / r^2
#pragma unroll
        for (int c = 0; c < RC; ++c)
            if (r0 + c < R) {
                const float4 v = sdd[(size_t)g * R + r0 + c];
                wr[c] = {v.x, v.y};
                wi[c] = {v.z, v.w};
            }
    }
    // the first warp loads the next tile's sources into registers while the tile runs
    float4 na, nb, nc, ns[RC];
    auto fetch = [&](int j0) {
        const int cnt = min(DFL_S, jhi - j0);
        if (lane < cnt) {
            const int g = bj.start + j0 + lane;
            na = pa[g]; nb = pb[g]; nc = pc[g];
#pragma unroll
            for (int c = 0; c < RC; ++c)
                ns[c] = (r0 + c < R) ? sdd[(size_t)g * R + r0 + c] : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {                                           // far, zero density: contributes 0 both ways
            na = make_float4(-1e5f - lane, -1e5f, -1e5f, 0.f);
            nb = nc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < RC; ++c) ns[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto stage = [&](DflTile<RC> &T) {
        T.a[lane] = na; T.b[lane] = nb; T.c[lane] = nc;
#pragma unroll
        for (int c = 0; c < RC; ++c) T.sig[lane][c] = ns[c];
    };
    if (warp == 0) {
        fetch(jlo);
        stage(s_tile[0]);
        if (jlo + DFL_S < jhi) fetch(jlo + DFL_S);
    }
    const bool warp_live = warp * 32 < bi.count;
    int buf = 0;
    for (int j0 = jlo; j0 < jhi; j0 += DFL_S, buf ^= 1) {
        const int cnt = min(DFL_S, jhi - j0);
        __syncthreads();                                   // tile j0 staged; the other buffer is free
        if (warp == 0 && j0 + DFL_S < jhi) {
            stage(s_tile[buf ^ 1]);
            if (j0 + 2 * DFL_S < jhi) fetch(j0 + 2 * DFL_S);
        }
        if (!warp_live) continue;
        const DflTile<RC> &T = s_tile[buf];
        dd asr[RC], asi[RC];
#pragma unroll
        for (int c = 0; c < RC; ++c) asr[c] = asi[c] = {0.f, 0.f};
        for (int s = st0; s < st1; ++s) {
            const int q = (lane + s) & (DFL_S - 1);
            const float4 A4 = T.a[q], B4 = T.b[q], C4 = T.c[q];
            const DflGeom G = dfl_geom<0>(tx, ty, tz, A4, B4, dd{0.f, 0.f}, s_tab, K);
            dd g1r, g1i, g2r, g2i;
            // i <- j: normal of source j
            dfl_kernel_value(G, dfl_projection({A4.w, B4.w}, {C4.x, C4.z}, {C4.y, C4.w}, G), K, g1r, g1i);
            // j <- i: normal of target i, d reversed
            dfl_kernel_value(G, dfl_projection(mx, my, mz, G), K, g2r, g2i);
#pragma unroll
            for (int c = 0; c < RC; ++c) {
                const float4 S = T.sig[q][c];
                const dd sr = {S.x, S.y}, si = {S.z, S.w};
                atr[c] = add(atr[c], sub(mul(g1r, sr), mul(g1i, si)));
                ati[c] = add(ati[c], add(mul(g1r, si), mul(g1i, sr)));
                asr[c] = add(asr[c], sub(mul(g2r, wr[c]), mul(g2i, wi[c])));
                asi[c] = add(asi[c], add(mul(g2r, wi[c]), mul(g2i, wr[c])));
            }
#pragma unroll
            for (int c = 0; c < RC; ++c) {
                const int from = (lane + 1) & 31;
                asr[c].h = __shfl_sync(0xffffffffu, asr[c].h, from);
                asr[c].l = __shfl_sync(0xffffffffu, asr[c].l, from);
                asi[c].h = __shfl_sync(0xffffffffu, asi[c].h, from);
                asi[c].l = __shfl_sync(0xffffffffu, asi[c].l, from);
            }
        }
#pragma unroll
        for (int c = 0; c < RC; ++c) { atr[c] = norm(atr[c]); ati[c] = norm(ati[c]); }
        // after the last step lane l holds this warp's sum for source (l + st1) mod 32:
        // straight into y
        const int src = (lane + st1) & (DFL_S - 1);
        if (src < cnt) {
#pragma unroll
            for (int c = 0; c < RC; ++c)
                if (r0 + c < R) {
                    double2 *o = y + (size_t)(bj.start + j0 + src) * R + r0 + c;
                    atomicAdd(&o->x, value(asr[c]) * scale[c]);
                    atomicAdd(&o->y, value(asi[c]) * scale[c]);
                }
        }
    }
    if (live) {
#pragma unroll
        for (int c = 0; c < RC; ++c)
            if (r0 + c < R) {
                double2 *o = y + (size_t)(bi.start + tid) * R + r0 + c;
                atomicAdd(&o->x, value(atr[c]) * scale[c]);
                atomicAdd(&o->y, value(ati[c]) * scale[c]);
            }
    }
}

// ---------------------------------------------------------------- one-directional kernel

// For several right-hand sides: one CTA per (TargetBlock part, chunk of RC right-hand sides,
// source chunk); a CTA of DFL_NT threads owns DFL_NT targets of a 512-target block, one per
// thread, each with a grid of its own per tile.  The source chunks divide the sources outside
// the block's own body, so all CTAs have equal work.  Per ordered pair the geometry,
// e^{ikr} and the kernel value are formed once and serve the RC right-hand sides, so wide
// chunks repeat the pair work least; the tile sums (4 RC registers) leave the running sums
// no registers: they stay in shared memory and are touched once per tile.  Source chunks
// write partial sums that a second kernel adds in a fixed order, so the result is
// bit-reproducible.
template <int RC, bool GRID>
__global__ void __launch_bounds__(DFL_NT, RC >= 32 ? 1 : 2)
nbody_dfl_kernel(const TargetBlock *__restrict__ blocks, int N, int R, int chunk, const float4 *__restrict__ pa,
                 const float4 *__restrict__ pb, const float4 *__restrict__ pc, const float2 *__restrict__ pw,
                 const float4 *__restrict__ sdd,
                 const int *__restrict__ key, const float4 *__restrict__ tab, DflConst K, double2 *__restrict__ y,
                 size_t split_stride)
{
    extern __shared__ float4 dfl_smem[];
    float4 *s_tab = dfl_smem;                              // DFL_TAB
    float4 *s_sig = s_tab + DFL_TAB;                       // DFL_S x RC
    float4 *s_a = s_sig + DFL_S * RC, *s_b = s_a + DFL_S, *s_c = s_b + DFL_S;
    float4 *s_run = s_c + DFL_S;                           // GRID: RC x DFL_NT running sums (re.hi, re.lo, im.hi, im.lo)
    __shared__ float2 s_w[DFL_S];
    __shared__ float s_wmax;
    __shared__ float4 s_ball;
    __shared__ int s_bits[2][RC];                          // largest high part of a tile's sigma', per column
    constexpr int LOADS = (DFL_S * RC + DFL_NT - 1) / DFL_NT;
    constexpr int PARTS = DFL_T / DFL_NT;
    const TargetBlock tb = blocks[blockIdx.x / PARTS];
    const int t0 = (blockIdx.x % PARTS) * DFL_NT;
    if (t0 >= tb.count) return;
    const int r0 = blockIdx.y * RC;
    const int tid = threadIdx.x, lane = tid & 31;
    for (int q = tid; q < DFL_TAB; q += DFL_NT) s_tab[q] = tab[q];
    const int g0 = tb.start + min(t0 + tid, tb.count - 1);
    const float4 TA = pa[g0], TB = pb[g0];
    const dd tx = {TA.x, TB.x}, ty = {TA.y, TB.y}, tz = {TA.z, TB.z};
    DflAcc ar[RC], ai[RC];                                 // GRID: the tile's sums
    dd zr[RC], zi[RC];                                     // else the running sums
#pragma unroll
    for (int c = 0; c < RC; ++c) {
        ar[c] = ai[c] = {0u, 0.f};
        zr[c] = zi[c] = {0.f, 0.f};
        if (GRID) s_run[c * DFL_NT + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (tid < 2 * RC) s_bits[tid / RC][tid % RC] = 0;
    // sources outside the own body, counted without it
    const int own = tb.excl_hi - tb.excl_lo;
    const int c0 = blockIdx.z * chunk, c1 = min(N - own, c0 + chunk);
    int buf = 0;
    for (int j0 = c0; j0 < c1; j0 += DFL_S, buf ^= 1) {
        const int cnt = min(DFL_S, c1 - j0);
        __syncthreads();
        if (tid < 32) {
            const int j = j0 + lane, g = j < tb.excl_lo ? j : j + own;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lane < cnt) {
                a = pa[g];
                s_a[lane] = a;
                s_b[lane] = pb[g];
                s_c[lane] = pc[g];
            }
            if (GRID) {
                const float2 w = lane < cnt ? pw[g] : make_float2(0.f, 0.f);
                s_w[lane] = w;
                const float4 ball = dfl_ball(a, lane < cnt, cnt);
                const int wm = __reduce_max_sync(0xffffffffu, __float_as_int(w.x));
                if (lane == 0) {
                    s_ball = ball;
                    s_wmax = __int_as_float(wm);
                }
            }
        }
        float4 v[LOADS];
#pragma unroll
        for (int u = 0; u < LOADS; ++u) {
            const int e = tid + u * DFL_NT, q = e / RC, c = e % RC, j = j0 + q, g = j < tb.excl_lo ? j : j + own;
            v[u] = (q < cnt && r0 + c < R) ? sdd[(size_t)g * R + r0 + c] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (GRID && q < cnt) atomicMax(&s_bits[buf][c], dfl_bits(v[u]));
        }
        if (GRID) {
            if (tid < RC) s_bits[buf ^ 1][tid] = 0;        // for the next tile
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < LOADS; ++u) {                  // GRID: scaled up to 1, column by column
            const int e = tid + u * DFL_NT;
            if (e < cnt * RC) s_sig[e] = GRID ? dfl_times(v[u], dfl_up(s_bits[buf][e % RC])) : v[u];
        }
        __syncthreads();
        const float fine =
            GRID ? dfl_fine(fmaxf(dfl_rmin(tx, ty, tz, s_ball, s_a, s_b, cnt), 0.f), K.kbound, s_wmax) : 0.f;
        unsigned corr = 0;                                 // the mantissas of the grids in the sums
        for (int jj = 0; jj < cnt; ++jj) {
            const float4 A4 = s_a[jj], B4 = s_b[jj], C4 = s_c[jj];
            const dd w = GRID ? dd{s_w[jj].x, s_w[jj].y} : dd{0.f, 0.f};
            const DflGeom G = dfl_geom<GRID>(tx, ty, tz, A4, B4, w, s_tab, K);
            dd gr, gi;
            dfl_kernel_value(G, dfl_projection({A4.w, B4.w}, {C4.x, C4.z}, {C4.y, C4.w}, G), K, gr, gi);
            if (GRID) {
                const DflGrid grid = dfl_grid(fmaxf(fabsf(gr.h), fabsf(gi.h)), fine);
                corr += __float_as_uint(grid.m) * grid.mult;
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    const float4 S = s_sig[jj * RC + c];
                    dfl_mac2(ar[c], gr, {S.x, S.y}, neg(gi), {S.z, S.w}, grid);
                    dfl_mac2(ai[c], gr, {S.z, S.w}, gi, {S.x, S.y}, grid);
                }
                if ((jj & 3) == 3) {
#pragma unroll
                    for (int c = 0; c < RC; ++c) {
                        dfl_carry(ar[c], fine);
                        dfl_carry(ai[c], fine);
                    }
                }
            } else {
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    const float4 S = s_sig[jj * RC + c];
                    const dd sr = {S.x, S.y}, si = {S.z, S.w};
                    zr[c] = add(zr[c], sub(mul(gr, sr), mul(gi, si)));
                    zi[c] = add(zi[c], add(mul(gr, si), mul(gi, sr)));
                }
            }
        }
        const float ulp = dfl_ulp_of(fine);
#pragma unroll
        for (int c = 0; c < RC; ++c) {
            if (GRID) {
                const float4 run = s_run[c * DFL_NT + tid];
                const float down = dfl_down(s_bits[buf][c]);
                const dd a = dfl_flush({run.x, run.y}, ar[c], corr, ulp, down),
                         b = dfl_flush({run.z, run.w}, ai[c], corr, ulp, down);
                s_run[c * DFL_NT + tid] = make_float4(a.h, a.l, b.h, b.l);
            } else {
                zr[c] = norm(zr[c]);
                zi[c] = norm(zi[c]);
            }
        }
    }
    if (t0 + tid < tb.count) {
        double2 *yo = y + blockIdx.z * split_stride;
#pragma unroll
        for (int c = 0; c < RC; ++c)
            if (r0 + c < R) {
                const float4 run = GRID ? s_run[c * DFL_NT + tid] : make_float4(zr[c].h, zr[c].l, zi[c].h, zi[c].l);
                const double sc = sigma_pow2(sigma_exponent(key[r0 + c]));
                yo[(size_t)(tb.start + t0 + tid) * R + r0 + c] =
                    make_double2(((double)run.x + (double)run.y) * sc, ((double)run.z + (double)run.w) * sc);
            }
    }
}

__global__ void dfl_split_reduce_kernel(size_t n, int nsplit, const double2 *__restrict__ part,
                                        double2 *__restrict__ y)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    double sx = 0.0, sy = 0.0;
    for (int s = 0; s < nsplit; ++s) {
        const double2 v = part[s * n + e];
        sx += v.x;
        sy += v.y;
    }
    y[e] = make_double2(sx, sy);
}

hzb_status dfl_split_reduce(hzb_ctx *c, size_t n, int nsplit, const double2 *part, double2 *y)
{
    dfl_split_reduce_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(n, nsplit, part, y);
    return check_cuda(c, cudaGetLastError(), "dfl_split_reduce_kernel");
}

// scaled node arrays and the table of cos/sin(2 pi m / 1024), high parts plus 3 on the grid of
// ulp(3), built once per context
hzb_status ensure_dfl(hzb_ctx *c)
{
    if (c->dfltab_ready) return HZB_OK;
    const size_t N = (size_t)c->N;
    if (check_cuda(c, c->dfltab.ensure(DFL_TAB), "alloc table") || check_cuda(c, c->dla.ensure(N), "alloc nodes") ||
        check_cuda(c, c->dlb.ensure(N), "alloc nodes") || check_cuda(c, c->dlc.ensure(N), "alloc nodes") ||
        check_cuda(c, c->dlw.ensure(N), "alloc nodes"))
        return HZB_ENOMEM;
    std::vector<float4> tab(DFL_TAB);
    for (int q = 0; q < DFL_TAB; ++q) {
        const long double a = 2.0L * 3.14159265358979323846264338327950288L * q / DFL_TAB;
        const double cv = (double)cosl(a), sv = (double)sinl(a);
        const float ch = (float)(cv + 3.0), sh = (float)(sv + 3.0);
        tab[q] = make_float4(ch, (float)(cv - ((double)ch - 3.0)), sh, (float)(sv - ((double)sh - 3.0)));
    }
    dfl_nodes_kernel<<<(unsigned)((N + 255) / 256), 256, 0, c->stream>>>(
        c->N, c->pos64.ptr, c->nrm64.ptr, make_double3(c->center[0], c->center[1], c->center[2]),
        c->k > 0.0 ? c->k / (2.0 * M_PI) : 1.0, c->dla.ptr, c->dlb.ptr, c->dlc.ptr, c->dlw.ptr);
    if (check_cuda(c, cudaGetLastError(), "dfl_nodes_kernel") ||
        check_cuda(c, cudaMemcpyAsync(c->dfltab.ptr, tab.data(), DFL_TAB * sizeof(float4), cudaMemcpyHostToDevice,
                                      c->stream), "copy table") ||
        check_cuda(c, cudaStreamSynchronize(c->stream), "table"))
        return HZB_ECUDA;
    c->dfltab_ready = true;
    return HZB_OK;
}

static dd dd_of(double v)
{
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

DflConst dfl_constants(const hzb_ctx *c)
{
    DflConst K;
    const double s = c->k > 0.0 ? c->k / (2.0 * M_PI) : 1.0, eta = c->eta / s;
    K.kappa = dd_of(c->k > 0.0 ? 2.0 * M_PI : 0.0);
    K.kbound = (float)((2.0 * M_PI + std::fabs(eta)) * 1.0001);
    int e;
    std::frexp(K.kbound, &e);                             // kbound < 2^e
    K.mb = (float)std::ldexp(1.5, e + 1);
    K.eta_m = (float)(eta + (double)K.mb);
    K.eta_r = (float)(eta - ((double)K.eta_m - (double)K.mb));
    K.no_phase = c->k > 0.0 ? 0 : 1;
    return K;
}

// key[r] of every column (sigma_scale.cuh) of c0 w_j sigma_{j,r} (weighted) or c0 sigma_{j,r}
hzb_status sigma_keys(hzb_ctx *c, int R, const double2 *sigma, double c0, int weighted, int *key)
{
    const size_t n = (size_t)c->N * R;
    if (check_cuda(c, cudaMemsetAsync(key, 0, R * sizeof(int), c->stream), "clear scales")) return HZB_ECUDA;
    const unsigned nb = (unsigned)std::min<size_t>((n + 2047) / 2048, 608);
    dfl_sigma_max_kernel<<<dim3(nb, (R + 255) / 256), 256, 0, c->stream>>>(c->N, R, c->pos64.ptr, sigma, c0, weighted,
                                                                           key);
    c->launches++;
    return check_cuda(c, cudaGetLastError(), "dfl_sigma_max_kernel");
}

// the densities of a call: weighted, scaled to below one per right-hand side, split
static hzb_status dfl_densities(hzb_ctx *c, int R, const double2 *sigma, int weighted)
{
    const size_t n = (size_t)c->N * R;
    if (check_cuda(c, c->dlsig.ensure(n), "alloc split densities") || check_cuda(c, c->dlkey.ensure(R), "alloc scales"))
        return HZB_ENOMEM;
    const double s = c->k > 0.0 ? c->k / (2.0 * M_PI) : 1.0, c0 = s * s / (4.0 * M_PI);
    if (n <= DFL_SIG_SMALL && R <= 64) {
        dfl_sigma_small_kernel<<<1, 1024, 0, c->stream>>>((int)n, R, c->pos64.ptr, sigma, c0, weighted,
                                                          c->dlkey.ptr, c->dlsig.ptr);
        c->launches += 1;
    } else {
        hzb_status st = sigma_keys(c, R, sigma, c0, weighted, c->dlkey.ptr);
        if (st) return st;
        dfl_sigma_split_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(n, R, c->pos64.ptr, sigma, c0,
                                                                                   weighted, c->dlkey.ptr, c->dlsig.ptr);
        c->launches += 1;
    }
    return check_cuda(c, cudaGetLastError(), "dfl_sigma_kernel");
}

// right-hand sides per CTA of the one-directional kernel
static int dfl_rc(int R) { return R == 1 ? 1 : (R <= 4 ? 4 : (R <= 8 ? 8 : (R <= 16 ? 16 : 32))); }

// Source chunks of the one-directional kernel: between six and twelve CTAs per resident
// place, the number whose last wave is fullest.
static int dfl_nsplit(hzb_ctx *c, int R, int nb)
{
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->opt.device);
    const int rc = dfl_rc(R);
    const long long places = (long long)sms * (rc >= 32 ? 1 : 2);
    const long long ctas = std::max<long long>(1, (long long)nb * (DFL_T / DFL_NT) * ((R + rc - 1) / rc));
    const long long lo = std::max<long long>(1, 6 * places / ctas), hi = std::max<long long>(1, 12 * places / ctas);
    long long best = std::min<long long>(lo, 64);
    double fill = 0.0;
    for (long long ns = best; ns <= std::min<long long>(hi, 64); ++ns) {
        const double waves = (double)(ns * ctas) / places, f = waves / std::ceil(waves);
        if (f > fill + 0.005) { fill = f; best = ns; }
    }
    return (int)best;
}

// the most sources that any target has: those outside the smallest body
static int dfl_sources(const hzb_ctx *c)
{
    long long n = 1;
    for (const BodyRec &b : c->bodies) n = std::max<long long>(n, c->N - b.n_nodes);
    for (const hzb_ctx::RShape &rs : c->rshapes) n = std::max<long long>(n, c->N - rs.k);
    return (int)n;
}

// Up to two right-hand sides the pair-symmetric kernel is the faster (4.10 against 5.44 ms at
// R = 1, 5.30 against 7.77 at R = 2, 29,280 unknowns), from three on the one-directional one
// (10.5 against 8.6 ms at R = 4), but for short sums, where the launch counts (432 unknowns,
// R = 4: 33 against 42 us).
bool dfl_symmetric(const hzb_ctx *c, int R) { return R <= 2 || (R <= 4 && dfl_sources(c) < DFL_GRID_MIN); }

// one-directional lean double-float sum (R right-hand sides in chunks of 1, 4, 8, 16 or
// 32, source chunks for occupancy, added in a fixed order)
hzb_status interbody_dfl(hzb_ctx *c, int R, const double2 *sigma, double2 *y)
{
    const int N = (int)c->N;
    const int rc = dfl_rc(R);
    const int nb = c->n_tblocks;
    const int nsrc = dfl_sources(c);
    // at R <= 4 the sums are a third of the work and the grid's upkeep eats what it saves
    const bool grid = nsrc >= DFL_GRID_MIN && rc >= 8;
    hzb_status st = ensure_dfl(c);
    if (st || (st = dfl_densities(c, R, sigma, grid ? 0 : 1))) return st;
    int nsplit = dfl_nsplit(c, R, nb);
    int chunk = (nsrc + nsplit - 1) / nsplit;
    chunk = ((chunk + DFL_S - 1) / DFL_S) * DFL_S;
    nsplit = (nsrc + chunk - 1) / chunk;
    const size_t n = (size_t)N * R;
    double2 *out = y;
    if (nsplit > 1) {
        if (check_cuda(c, c->nb_part64.ensure(n * nsplit), "alloc partial sums")) return HZB_ENOMEM;
        out = c->nb_part64.ptr;
    }
    const DflConst K = dfl_constants(c);
    c->interbody_calls++;
    c->launches += (nsplit > 1) ? 2 : 1;
    const int slot = prof_begin(c, 2);
    const size_t smem = sizeof(float4) * ((size_t)DFL_TAB + (grid ? (size_t)rc * DFL_NT : 0) + (size_t)DFL_S * (rc + 3));
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kern) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return;
        dim3 g((unsigned)(nb * (DFL_T / DFL_NT)), (R + rc - 1) / rc, nsplit);
        kern<<<g, DFL_NT, smem, c->stream>>>(c->tblocks.ptr, N, R, chunk, c->dla.ptr, c->dlb.ptr, c->dlc.ptr,
                                             c->dlw.ptr, c->dlsig.ptr, c->dlkey.ptr, c->dfltab.ptr, K, out, n);
        e = cudaGetLastError();
    };
    switch (rc) {
    case 1: launch(nbody_dfl_kernel<1, false>); break;
    case 4: launch(nbody_dfl_kernel<4, false>); break;
    case 8: grid ? launch(nbody_dfl_kernel<8, true>) : launch(nbody_dfl_kernel<8, false>); break;
    case 16: grid ? launch(nbody_dfl_kernel<16, true>) : launch(nbody_dfl_kernel<16, false>); break;
    default: grid ? launch(nbody_dfl_kernel<32, true>) : launch(nbody_dfl_kernel<32, false>); break;
    }
    if (nsplit > 1) dfl_split_reduce_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c->stream>>>(n, nsplit, out, y);
    if (e == cudaSuccess) e = cudaGetLastError();
    prof_end(c, slot);
    return check_cuda(c, e, "nbody_dfl_kernel");
}

// pair-symmetric lean double-float sum
hzb_status interbody_dfl_sym(hzb_ctx *c, int R, const double2 *sigma, double2 *y)
{
    if (c->capturing && (c->n_blockpairs == 0 || !c->dfltab_ready))
        return fail(c, HZB_ESTATE, "block pairs or table not built before capture");
    hzb_status st = ensure_block_pairs(c);
    if (st) return st;
    if ((st = ensure_dfl(c))) return st;
    const size_t n = (size_t)c->N * R;
    if (check_cuda(c, cudaMemsetAsync(y, 0, n * sizeof(double2), c->stream), "zero y")) return HZB_ECUDA;
    c->interbody_calls++;
    if (c->n_blockpairs < 0) return HZB_OK;
    if (c->n_blockpairs > 0x7fffffffLL) return fail(c, HZB_EINVAL, "too many block pairs for one launch");
    if ((st = dfl_densities(c, R, sigma, 1))) return st;
    c->launches += 1;
    const DflConst K = dfl_constants(c);
    const int slot = prof_begin(c, 2);
    const int rc = (R == 1) ? 1 : 2;
    const SymSplit sp = sym_split(c, (R + rc - 1) / rc, 1);
    dim3 g((unsigned)c->n_blockpairs, (R + rc - 1) / rc, sp.nz);
    auto launch = [&](auto kern) {
        kern<<<g, DFL_T, 0, c->stream>>>(c->blockpairs.ptr, c->tblocks.ptr, R, c->dla.ptr, c->dlb.ptr, c->dlc.ptr,
                                         c->dlsig.ptr, c->dlkey.ptr, c->dfltab.ptr, K, y, sp);
    };
    if (rc == 1) launch(nbody_dfl_sym_kernel<1>);
    else launch(nbody_dfl_sym_kernel<2>);
    cudaError_t e = cudaGetLastError();
    prof_end(c, slot);
    return check_cuda(c, e, "nbody_dfl_sym_kernel");
}

}  // namespace hzb
