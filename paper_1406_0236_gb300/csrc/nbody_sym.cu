// FP64 inter-body sum y = B sigma (Sec. 3.3, Eq. (nystromnaive)) with each unordered
// pair of nodes on different bodies evaluated once for both directions.
//
// For nodes i, j with d = x_i - x_j, r = |d|:
//     w_j K(x_i, x_j) = w_j / (4 pi) e^{ikr} [ n_j.d / r^3 - i (k n_j.d / r^2 + eta / r) ]
//     w_i K(x_j, x_i) = w_i / (4 pi) e^{ikr} [-n_i.d / r^3 - i (-k n_i.d / r^2 + eta / r) ]
// share d, r, 1/r and e^{ikr}, which are two thirds of the FP64 work of a pair; the
// two directions differ only in the normal projection.  About 25 FP64 operations
// per ordered pair instead of 41 for the one-directional kernel (nbody64_kernel).
//
// Work: one CTA per unordered pair of TargetBlocks (I, J), I < J, on different
// bodies (grid y: chunks of RC right-hand sides).  Thread t owns target i = I.start + t;
// sources of J come in tiles of 32.  Inside a warp the 32 x 32 pairs of a tile run in
// 32 steps: at step s lane l takes source (l + s) mod 32, adds the i <- j term to its
// own sum and the j <- i term to a rotating sum that then moves to lane l - 1, so each
// source's partial sum visits every lane once and no two lanes touch the same source
// at a step.  The warps' partial sums of a tile are added in a fixed order in shared
// memory.  On small geometries several CTAs share a block pair (sym_split).  Both directions
// reach y through FP64 atomic adds (y is zeroed first), so the order of the additions into one y
// entry varies between runs: the result is reproducible to rounding, not bit for bit.
#include <algorithm>
#include <cmath>
#include <vector>

#include "f32x2.cuh"
#include "fp64_pair.cuh"
#include "hzb_internal.h"
#include "kernel_math.cuh"

namespace hzb {

static const int SYM_T = 512;        // targets per CTA = TargetBlock size
static const int SYM_S = 32;         // sources per tile (one per lane)

// Constants of the FP64 kernel: phase in table units, normals times nf, densities times wf.
struct SymConst {
    double kt, ik, k, eta, nf, wf;
};

// Whether eta and k leave the scaled forms of the two kernels in range (else GEN).
bool sym_scaled(const hzb_ctx *c)
{
    const double q = std::fabs(c->eta) / c->k;
    return c->k >= 1e-6 && q >= 1e-6 && q <= 1e6;
}

// This CTA's part of its block pair (SymSplit): sources [jlo, jhi) of J and rotation
// steps [st0, st1) of each of their tiles.
__device__ __forceinline__ void sym_range(const SymSplit &sp, int nj, int &jlo, int &jhi, int &st0, int &st1)
{
    const int zj = blockIdx.z / sp.nstep, zs = blockIdx.z % sp.nstep;
    jlo = zj * sp.jchunk;
    jhi = min(nj, jlo + sp.jchunk);
    st0 = zs * (SYM_S / sp.nstep);
    st1 = st0 + SYM_S / sp.nstep;
}

// With E = e^{ikr} / r = a + i b the pair's two kernel values are, up to the common factor eta,
//     (n~.d) P + b - i a,   P = (1/r) [(a v + b) + i (b v - a)],  v = 1 / (k r),
// for the normal n~ = (k / eta) n of the source side: P serves both directions, the single
// layer's part is E itself, and the factor goes into the densities.  50 FP64 operations per
// unordered pair with one right-hand side (55 with the two layers formed per direction: 31.4 ->
// 28.3 ms at 29,280 unknowns), 92 % of the FP64 pipe.  GEN: any k and eta, P and E with
// their factors (k, eta) in place.
template <int RC, bool GEN>
__global__ void __launch_bounds__(SYM_T, 1)
nbody64_sym_kernel(const int2 *__restrict__ pairs, const TargetBlock *__restrict__ blocks, int R,
                   const double4 *__restrict__ pos, const double4 *__restrict__ nrm,
                   const double2 *__restrict__ sigma, const double2 *__restrict__ sctab, SymConst K,
                   double2 *__restrict__ y, SymSplit sp)
{
    __shared__ double4 s_p[SYM_S];               // x, y, z, w
    __shared__ double4 s_n[SYM_S];               // nx, ny, nz
    __shared__ double2 s_w[SYM_S][RC];           // w_j sigma_j / (4 pi)
    __shared__ double2 s_red[SYM_T / 32][RC][SYM_S];
    const int2 pr = pairs[blockIdx.x];
    const TargetBlock bi = blocks[pr.x], bj = blocks[pr.y];
    int jlo, jhi, st0, st1;                      // this CTA's sources of J and rotation steps
    sym_range(sp, bj.count, jlo, jhi, st0, st1);
    if (jlo >= jhi) return;
    const int r0 = blockIdx.y * RC;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool live = tid < bi.count;
    // own target: position, normal, weighted densities (zero for padding threads)
    double tx = 1e6 + tid, ty = 1e6, tz = 1e6, mx = 0.0, my = 0.0, mz = 0.0;
    double2 wi[RC], acc_t[RC];
    if (live) {
        const double4 p = pos[bi.start + tid], n = nrm[bi.start + tid];
        tx = p.x; ty = p.y; tz = p.z;
        mx = -K.nf * n.x; my = -K.nf * n.y; mz = -K.nf * n.z;         // negated: d is reversed for j <- i
        const double wq = p.w * K.wf;
#pragma unroll
        for (int c = 0; c < RC; ++c) {
            const double2 v = (r0 + c < R) ? sigma[(size_t)(bi.start + tid) * R + r0 + c] : make_double2(0.0, 0.0);
            wi[c] = make_double2(v.x * wq, v.y * wq);
        }
    } else {
#pragma unroll
        for (int c = 0; c < RC; ++c) wi[c] = make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int c = 0; c < RC; ++c) acc_t[c] = make_double2(0.0, 0.0);
    const bool warp_live = warp * 32 < bi.count;
    for (int j0 = jlo; j0 < jhi; j0 += SYM_S) {
        const int cnt = min(SYM_S, jhi - j0);
        __syncthreads();
        if (tid < SYM_S) {
            if (tid < cnt) {
                const double4 p = pos[bj.start + j0 + tid];
                s_p[tid] = p;
                const double4 n = nrm[bj.start + j0 + tid];
                s_n[tid] = make_double4(K.nf * n.x, K.nf * n.y, K.nf * n.z, 0.0);
                const double wq = p.w * K.wf;
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    const double2 v =
                        (r0 + c < R) ? sigma[(size_t)(bj.start + j0 + tid) * R + r0 + c] : make_double2(0.0, 0.0);
                    s_w[tid][c] = make_double2(v.x * wq, v.y * wq);
                }
            } else {                                   // far, zero density: contributes 0 both ways
                s_p[tid] = make_double4(-1e6 - tid, -1e6, -1e6, 0.0);
                s_n[tid] = make_double4(0.0, 0.0, 0.0, 0.0);
#pragma unroll
                for (int c = 0; c < RC; ++c) s_w[tid][c] = make_double2(0.0, 0.0);
            }
        }
        __syncthreads();
        double2 acc_s[RC];
#pragma unroll
        for (int c = 0; c < RC; ++c) acc_s[c] = make_double2(0.0, 0.0);
        if (warp_live) {
#pragma unroll 2
            for (int s = st0; s < st1; ++s) {
                const int q = (lane + s) & (SYM_S - 1);
                const double4 p = s_p[q];
                const double4 n = s_n[q];
                const double dx = tx - p.x, dy = ty - p.y, dz = tz - p.z;
                const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                const double ir = rsqrt_fp64(r2);
                double sn, cs;
                cis_turns((r2 * ir) * K.kt, sctab, cs, sn);
                const double ea = cs * ir, eb = sn * ir;
                const double v = GEN ? ir : ir * K.ik;
                const double pr = ir * fma(ea, v, GEN ? K.k * eb : eb);
                const double pn = ir * fma(-eb, v, GEN ? K.k * ea : ea);        // -Im P
                const double qb = GEN ? K.eta * eb : eb, qa = GEN ? K.eta * ea : ea;
                // i <- j: normal of source j; g1n = -Im
                const double X1 = fma(n.x, dx, fma(n.y, dy, n.z * dz));
                const double g1r = fma(X1, pr, qb), g1n = fma(X1, pn, qa);
                // j <- i: normal of target i, d reversed
                const double X2 = fma(mx, dx, fma(my, dy, mz * dz));
                const double g2r = fma(X2, pr, qb), g2n = fma(X2, pn, qa);
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    const double2 wj = s_w[q][c];
                    acc_t[c].x = fma(g1r, wj.x, fma(g1n, wj.y, acc_t[c].x));
                    acc_t[c].y = fma(g1r, wj.y, fma(-g1n, wj.x, acc_t[c].y));
                    acc_s[c].x = fma(g2r, wi[c].x, fma(g2n, wi[c].y, acc_s[c].x));
                    acc_s[c].y = fma(g2r, wi[c].y, fma(-g2n, wi[c].x, acc_s[c].y));
                }
                // the rotating sum of source (l + s + 1) mod 32 comes from lane l + 1
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    acc_s[c].x = __shfl_sync(0xffffffffu, acc_s[c].x, (lane + 1) & 31);
                    acc_s[c].y = __shfl_sync(0xffffffffu, acc_s[c].y, (lane + 1) & 31);
                }
            }
        }
        // after the last step lane l holds the partial sum of source (l + st1) mod 32
#pragma unroll
        for (int c = 0; c < RC; ++c) s_red[warp][c][(lane + st1) & (SYM_S - 1)] = acc_s[c];
        __syncthreads();
        if (tid < SYM_S * RC) {
            const int src = tid & (SYM_S - 1), c = tid / SYM_S;
            if (src < cnt && r0 + c < R) {
                double sx = 0.0, sy = 0.0;
                for (int w = 0; w < SYM_T / 32; ++w) {
                    sx += s_red[w][c][src].x;
                    sy += s_red[w][c][src].y;
                }
                double2 *o = y + (size_t)(bj.start + j0 + src) * R + r0 + c;
                atomicAdd(&o->x, sx);
                atomicAdd(&o->y, sy);
            }
        }
    }
    if (live) {
#pragma unroll
        for (int c = 0; c < RC; ++c)
            if (r0 + c < R) {
                double2 *o = y + (size_t)(bi.start + tid) * R + r0 + c;
                atomicAdd(&o->x, acc_t[c].x);
                atomicAdd(&o->y, acc_t[c].y);
            }
    }
}

// FP32 version for the inner solve, with packed f32x2 pairs (f32x2.cuh): thread t
// owns TP pairs of targets (t + 2p NT, t + (2p + 1) NT), packed in the two halves of
// each register pair, and meets one source per step as above, so one f32x2
// instruction serves two unordered node pairs.  The rotating source sums keep the
// two halves apart and add them at the end of the tile.  Densities come pre-weighted
// in FP32 (weighted_sigma32), positions times k and normals times k / eta (rounded once from
// FP64, sym32_nodes_kernel), so that r is the phase and v = 1/r: the form of the FP64 kernel
// in 32 lane operations per unordered pair and right-hand side one, 36 before (36.9 ->
// 34.1 ms at 258,560 unknowns); e^{ikr} comes straight from the transcendental unit
// (its own argument scaling).  GEN as in the FP64 kernel, lengths and normals unscaled.
// One right-hand side with two packed target pairs per thread is held to 96 registers, five
// 128-thread CTAs per SM, with four steps unrolled: 64,640 unknowns 2.19 ms, against 2.27 for
// six CTAs at 80 registers and two steps, 2.23 for four CTAs, 2.22 for six and 2.41 for seven.
static constexpr int SYM32_MIN_BLOCKS = 5;
// STEPS = false: all 32 rotation steps, a constant trip count (2 % of the time at 258,560
// unknowns against the bounds of a split).
template <int RC, int TP, bool STEPS, bool GEN>
__global__ void __launch_bounds__(SYM_T / (2 * TP), (RC == 1 && TP == 2) ? SYM32_MIN_BLOCKS : 1)
nbody32_sym_kernel(const int2 *__restrict__ pairs, const TargetBlock *__restrict__ blocks, int R,
                   const float4 *__restrict__ pos, const float4 *__restrict__ nrm, const float2 *__restrict__ sw,
                   float k, float eta, double2 *__restrict__ y, SymSplit sp)
{
    constexpr int NT = SYM_T / (2 * TP);
    constexpr int NW = NT / 32;
    __shared__ float4 s_g0[SYM_S];               // x, y, z, nx
    __shared__ float2 s_g1[SYM_S];               // ny, nz
    __shared__ float2 s_w[SYM_S][RC];
    __shared__ float2 s_red[NW][RC][SYM_S];
    const int2 pr = pairs[blockIdx.x];
    const TargetBlock bi = blocks[pr.x], bj = blocks[pr.y];
    int jlo, jhi, st0, st1;                      // this CTA's sources of J and rotation steps
    sym_range(sp, bj.count, jlo, jhi, st0, st1);
    if (!STEPS) { st0 = 0; st1 = SYM_S; }
    if (jlo >= jhi) return;
    const int r0 = blockIdx.y * RC;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    f2x tx[TP], ty[TP], tz[TP], mx[TP], my[TP], mz[TP];      // target positions, negated normals
    f2x wr[TP][RC], wi[TP][RC], nwr[TP][RC], atx[TP][RC], aty[TP][RC];
#pragma unroll
    for (int p = 0; p < TP; ++p) {
        float4 P[2], Q[2];
        float2 V[2][RC];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = tid + (2 * p + h) * NT;
            const bool live = t < bi.count;
            P[h] = live ? pos[bi.start + t] : make_float4(1e5f + t, 1e5f, 1e5f, 0.f);
            Q[h] = live ? nrm[bi.start + t] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < RC; ++c)
                V[h][c] = (live && r0 + c < R) ? sw[(size_t)(bi.start + t) * R + r0 + c] : make_float2(0.f, 0.f);
        }
        tx[p] = f2_pack(P[0].x, P[1].x); ty[p] = f2_pack(P[0].y, P[1].y); tz[p] = f2_pack(P[0].z, P[1].z);
        mx[p] = f2_pack(-Q[0].x, -Q[1].x); my[p] = f2_pack(-Q[0].y, -Q[1].y); mz[p] = f2_pack(-Q[0].z, -Q[1].z);
#pragma unroll
        for (int c = 0; c < RC; ++c) {
            wr[p][c] = f2_pack(V[0][c].x, V[1][c].x);
            wi[p][c] = f2_pack(V[0][c].y, V[1][c].y);
            nwr[p][c] = f2_pack(-V[0][c].x, -V[1][c].x);
            atx[p][c] = aty[p][c] = 0ull;
        }
    }
    const bool warp_live = warp * 32 < bi.count;
    const f2x k2 = f2_splat(k), eta2 = f2_splat(eta);
    for (int j0 = jlo; j0 < jhi; j0 += SYM_S) {
        const int cnt = min(SYM_S, jhi - j0);
        __syncthreads();
        if (tid < SYM_S) {
            if (tid < cnt) {
                const float4 p = pos[bj.start + j0 + tid], n = nrm[bj.start + j0 + tid];
                s_g0[tid] = make_float4(p.x, p.y, p.z, n.x);
                s_g1[tid] = make_float2(n.y, n.z);
#pragma unroll
                for (int c = 0; c < RC; ++c)
                    s_w[tid][c] = (r0 + c < R) ? sw[(size_t)(bj.start + j0 + tid) * R + r0 + c] : make_float2(0.f, 0.f);
            } else {                                   // far, zero density: contributes 0 both ways
                s_g0[tid] = make_float4(-1e5f - tid, -1e5f, -1e5f, 0.f);
                s_g1[tid] = make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < RC; ++c) s_w[tid][c] = make_float2(0.f, 0.f);
            }
        }
        __syncthreads();
        f2x asx[RC], asy[RC];
#pragma unroll
        for (int c = 0; c < RC; ++c) asx[c] = asy[c] = 0ull;
        if (warp_live) {
#pragma unroll 4
            for (int s = st0; s < st1; ++s) {
                const int q = (lane + s) & (SYM_S - 1);
                const float4 g0 = s_g0[q];
                const float2 g1 = s_g1[q];
                const f2x sx = f2_splat(g0.x), sy = f2_splat(g0.y), sz = f2_splat(g0.z);
                const f2x snx = f2_splat(g0.w), sny = f2_splat(g1.x), snz = f2_splat(g1.y);
                f2x swr[RC], swi[RC], nswr[RC];
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    const float2 v = s_w[q][c];
                    swr[c] = f2_splat(v.x); swi[c] = f2_splat(v.y); nswr[c] = f2_splat(-v.x);
                }
#pragma unroll
                for (int p = 0; p < TP; ++p) {
                    const f2x dx = f2_sub(tx[p], sx), dy = f2_sub(ty[p], sy), dz = f2_sub(tz[p], sz);
                    const f2x r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
                    float r2a, r2b;
                    f2_unpack(r2, r2a, r2b);
                    const f2x ir = f2_pack(rsqrtf(r2a), rsqrtf(r2b));
                    const f2x kr = GEN ? f2_mul(f2_mul(r2, ir), k2) : f2_mul(r2, ir);
                    // e^{ikr}: the transcendental unit reduces the argument itself (its
                    // scaling to turns rounds like an explicit reduction would)
                    float kra, krb, sa, ca, sb, cb;
                    f2_unpack(kr, kra, krb);
                    __sincosf(kra, &sa, &ca);
                    __sincosf(krb, &sb, &cb);
                    const f2x ea = f2_mul(f2_pack(ca, cb), ir), eb = f2_mul(f2_pack(sa, sb), ir);
                    const f2x pr = f2_mul(ir, f2_fma(ea, ir, GEN ? f2_mul(k2, eb) : eb));
                    const f2x pn = f2_mul(ir, f2_fma(f2_neg(eb), ir, GEN ? f2_mul(k2, ea) : ea));     // -Im P
                    const f2x qb = GEN ? f2_mul(eta2, eb) : eb, qa = GEN ? f2_mul(eta2, ea) : ea;
                    // target <- source q; g1n = -Im
                    const f2x X1 = f2_fma(snx, dx, f2_fma(sny, dy, f2_mul(snz, dz)));
                    const f2x g1r = f2_fma(X1, pr, qb), g1n = f2_fma(X1, pn, qa);
                    // source q <- target, d reversed (the target normals are stored negated)
                    const f2x X2 = f2_fma(mx[p], dx, f2_fma(my[p], dy, f2_mul(mz[p], dz)));
                    const f2x g2r = f2_fma(X2, pr, qb), g2n = f2_fma(X2, pn, qa);
#pragma unroll
                    for (int c = 0; c < RC; ++c) {
                        atx[p][c] = f2_fma(g1r, swr[c], f2_fma(g1n, swi[c], atx[p][c]));
                        aty[p][c] = f2_fma(g1r, swi[c], f2_fma(g1n, nswr[c], aty[p][c]));
                        asx[c] = f2_fma(g2r, wr[p][c], f2_fma(g2n, wi[p][c], asx[c]));
                        asy[c] = f2_fma(g2r, wi[p][c], f2_fma(g2n, nwr[p][c], asy[c]));
                    }
                }
#pragma unroll
                for (int c = 0; c < RC; ++c) {
                    asx[c] = __shfl_sync(0xffffffffu, asx[c], (lane + 1) & 31);
                    asy[c] = __shfl_sync(0xffffffffu, asy[c], (lane + 1) & 31);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < RC; ++c) {
            float xa, xb, ya, yb;
            f2_unpack(asx[c], xa, xb);
            f2_unpack(asy[c], ya, yb);
            s_red[warp][c][(lane + st1) & (SYM_S - 1)] = make_float2(xa + xb, ya + yb);
        }
        __syncthreads();
        if (tid < SYM_S * RC) {
            const int src = tid & (SYM_S - 1), c = tid / SYM_S;
            if (src < cnt && r0 + c < R) {
                float sx = 0.f, sy = 0.f;
                for (int w = 0; w < NW; ++w) {
                    sx += s_red[w][c][src].x;
                    sy += s_red[w][c][src].y;
                }
                double2 *o = y + (size_t)(bj.start + j0 + src) * R + r0 + c;
                atomicAdd(&o->x, (double)sx);
                atomicAdd(&o->y, (double)sy);
            }
        }
    }
#pragma unroll
    for (int p = 0; p < TP; ++p)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = tid + (2 * p + h) * NT;
            if (t >= bi.count) continue;
#pragma unroll
            for (int c = 0; c < RC; ++c)
                if (r0 + c < R) {
                    float xa, xb, ya, yb;
                    f2_unpack(atx[p][c], xa, xb);
                    f2_unpack(aty[p][c], ya, yb);
                    double2 *o = y + (size_t)(bi.start + t) * R + r0 + c;
                    atomicAdd(&o->x, (double)(h ? xb : xa));
                    atomicAdd(&o->y, (double)(h ? yb : ya));
                }
        }
}

// A block pair per CTA leaves most of the chip idle on small geometries (two spheres of
// 4,100 nodes: 81 CTAs; 216 nodes: one), and a CTA of 512 x 512 pairs is a long last wave on
// middling ones.  So the source side is cut until there are about 16 CTAs per SM, down to
// one tile of 32 sources, and below `steps_below` per SM the rotation steps of a tile are shared
// out too.  Finer pieces cost more than they fill: every CTA adds its 512 target sums to y with
// FP64 atomics.  Before -> after, one right-hand side (FP64 / double-float / FP32 sums):
// 432 unknowns 787 / 139 / 61 -> 16 / 19 / 16 us each (the call itself); 8,200 unknowns 3,814 /
// 533 / 122 -> 1,672 / 263 / 39 us (at twice as many pieces 1,693 / 295 / 39); 29,280 unknowns
// 32.31 / 4.47 / 0.523 -> 31.41 / 4.37 / 0.455 ms; from 64,640 unknowns up nothing is cut.
// steps_below = 4, 2, 1, us: 1,350 unknowns on three bodies, FP64 85, 92, 112, double-float 66, 42,
// 38, FP32 30, 20, 17; 3,968 on two, R = 4: FP64 591, 648, 636, FP32 52, 36, 29, R = 1 double-float
// 99, 93, 84; 2,640 on eight: FP64 385, 451, 451, double-float 88, 94, 94, FP32 20, 21, 22.
SymSplit sym_split(hzb_ctx *c, int rhs_chunks, int steps_below)
{
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->opt.device);
    const long long have = c->n_blockpairs * rhs_chunks;
    SymSplit sp = {SYM_T, 1, 1};
    while (have * sp.nz < 16LL * sms && sp.jchunk > SYM_S) { sp.jchunk /= 2; sp.nz *= 2; }
    while (have * sp.nz < (long long)steps_below * sms && sp.nstep < 16) { sp.nstep *= 2; sp.nz *= 2; }
    return sp;
}

// Unordered pairs of target blocks on different bodies, built once per geometry.
hzb_status ensure_block_pairs(hzb_ctx *c)
{
    if (c->n_blockpairs > 0) return HZB_OK;
    std::vector<TargetBlock> tb(c->n_tblocks);
    if (check_cuda(c, cudaMemcpyAsync(tb.data(), c->tblocks.ptr, tb.size() * sizeof(TargetBlock),
                                      cudaMemcpyDeviceToHost, c->stream), "copy blocks") ||
        check_cuda(c, cudaStreamSynchronize(c->stream), "copy blocks"))
        return HZB_ECUDA;
    // the CTA's threads own the targets of pair.x and step through the sources of pair.y:
    // the larger block goes first, so a body's short last block is always the source side
    // (a short CTA) and never leaves most of a CTA's threads idle for a full pass
    std::vector<int2> pr;
    for (int i = 0; i < (int)tb.size(); ++i)
        for (int j = i + 1; j < (int)tb.size(); ++j)
            if (tb[i].excl_lo != tb[j].excl_lo)
                pr.push_back(tb[j].count > tb[i].count ? make_int2(j, i) : make_int2(i, j));
    if (pr.empty()) {
        c->n_blockpairs = -1;                   // one body: B = 0
        return HZB_OK;
    }
    if (check_cuda(c, c->blockpairs.ensure(pr.size()), "alloc block pairs")) return HZB_ENOMEM;
    if (check_cuda(c, cudaMemcpyAsync(c->blockpairs.ptr, pr.data(), pr.size() * sizeof(int2),
                                      cudaMemcpyHostToDevice, c->stream), "copy block pairs") ||
        check_cuda(c, cudaStreamSynchronize(c->stream), "copy block pairs"))
        return HZB_ECUDA;
    c->n_blockpairs = (long long)pr.size();
    return HZB_OK;
}

hzb_status interbody64_sym(hzb_ctx *c, int R, const double2 *sigma, double2 *y)
{
    if (!c->nodes_ready) return fail(c, HZB_ESTATE, "nodes not built");
    if (c->capturing && c->n_blockpairs == 0) return fail(c, HZB_ESTATE, "block pairs not built before capture");
    hzb_status st = ensure_sctab(c);
    if (st || (st = ensure_block_pairs(c))) return st;
    const size_t n = (size_t)c->N * R;
    if (check_cuda(c, cudaMemsetAsync(y, 0, n * sizeof(double2), c->stream), "zero y")) return HZB_ECUDA;
    c->interbody_calls++;
    if (c->n_blockpairs < 0) return HZB_OK;
    if (c->n_blockpairs > 0x7fffffffLL) return fail(c, HZB_EINVAL, "too many block pairs for one launch");
    c->launches += 1;
    const int slot = prof_begin(c, 0);
    const int rc = (R == 1) ? 1 : (R == 2 ? 2 : 4);
    const SymSplit sp = sym_split(c, (R + rc - 1) / rc, 4);
    dim3 g((unsigned)c->n_blockpairs, (R + rc - 1) / rc, sp.nz);
    const bool gen = !sym_scaled(c);
    const SymConst K = {c->k * (SC_N / (2.0 * M_PI)), gen ? 0.0 : 1.0 / c->k, c->k, c->eta,
                        gen ? 1.0 : c->k / c->eta, (gen ? 1.0 : c->eta) * HZB_INV4PI};
    auto launch = [&](auto kern) {
        kern<<<g, SYM_T, 0, c->stream>>>(c->blockpairs.ptr, c->tblocks.ptr, R, c->pos64.ptr, c->nrm64.ptr, sigma,
                                         c->sctab.ptr, K, y, sp);
    };
    if (rc == 1) gen ? launch(nbody64_sym_kernel<1, true>) : launch(nbody64_sym_kernel<1, false>);
    else if (rc == 2) gen ? launch(nbody64_sym_kernel<2, true>) : launch(nbody64_sym_kernel<2, false>);
    else gen ? launch(nbody64_sym_kernel<4, true>) : launch(nbody64_sym_kernel<4, false>);
    cudaError_t e = cudaGetLastError();
    prof_end(c, slot);
    return check_cuda(c, e, "nbody64_sym_kernel");
}

// positions relative to the centre and normals of the FP32 kernel, scaled (see there)
__global__ void sym32_nodes_kernel(long long N, const double4 *__restrict__ pos, const double4 *__restrict__ nrm,
                                   double3 o, double ps, double ns, float4 *__restrict__ p32, float4 *__restrict__ n32)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const double4 p = pos[i], n = nrm[i];
    p32[i] = make_float4((float)((p.x - o.x) * ps), (float)((p.y - o.y) * ps), (float)((p.z - o.z) * ps), 0.f);
    n32[i] = make_float4((float)(n.x * ns), (float)(n.y * ns), (float)(n.z * ns), 0.f);
}

hzb_status ensure_sym32(hzb_ctx *c)
{
    if (c->sym32_ready) return HZB_OK;
    if (c->capturing) return fail(c, HZB_ESTATE, "scaled nodes not built before capture");
    if (check_cuda(c, c->symn.ensure(2 * (size_t)c->N), "alloc scaled nodes")) return HZB_ENOMEM;
    const bool gen = !sym_scaled(c);
    sym32_nodes_kernel<<<(unsigned)((c->N + 255) / 256), 256, 0, c->stream>>>(
        c->N, c->pos64.ptr, c->nrm64.ptr, make_double3(c->center[0], c->center[1], c->center[2]), gen ? 1.0 : c->k,
        gen ? 1.0 : c->k / c->eta, c->symn.ptr, c->symn.ptr + c->N);
    if (check_cuda(c, cudaGetLastError(), "sym32_nodes_kernel")) return HZB_ECUDA;
    c->sym32_ready = true;
    return HZB_OK;
}

template <int RC, int TP>
static void launch_sym32(hzb_ctx *c, dim3 g, int R, const float2 *sw, double2 *y, SymSplit sp)
{
    auto launch = [&](auto kern) {
        kern<<<g, SYM_T / (2 * TP), 0, c->stream>>>(c->blockpairs.ptr, c->tblocks.ptr, R, c->symn.ptr, c->symn.ptr + c->N, sw,
                                                    (float)c->k, (float)c->eta, y, sp);
    };
    const bool gen = !sym_scaled(c);
    if (sp.nstep > 1) gen ? launch(nbody32_sym_kernel<RC, TP, true, true>) : launch(nbody32_sym_kernel<RC, TP, true, false>);
    else gen ? launch(nbody32_sym_kernel<RC, TP, false, true>) : launch(nbody32_sym_kernel<RC, TP, false, false>);
}

hzb_status interbody32_sym(hzb_ctx *c, int R, const double2 *sigma, double2 *y, int tp)
{
    if (!c->nodes_ready) return fail(c, HZB_ESTATE, "nodes not built");
    if (c->capturing && c->n_blockpairs == 0) return fail(c, HZB_ESTATE, "block pairs not built before capture");
    hzb_status st = ensure_block_pairs(c);
    if (st || (st = ensure_sym32(c))) return st;
    const size_t n = (size_t)c->N * R;
    if (check_cuda(c, cudaMemsetAsync(y, 0, n * sizeof(double2), c->stream), "zero y")) return HZB_ECUDA;
    c->interbody_calls++;
    if (c->n_blockpairs < 0) return HZB_OK;
    if (c->n_blockpairs > 0x7fffffffLL) return fail(c, HZB_EINVAL, "too many block pairs for one launch");
    const int slot = prof_begin(c, 1);
    const float2 *sw = weighted_sigma32(c, R, sigma, sym_scaled(c) ? c->k * c->eta : 1.0);
    if (!sw) return HZB_ENOMEM;
    c->launches += 1;
    const int rc = (R == 1) ? 1 : (R == 2 ? 2 : 4);
    const SymSplit sp = sym_split(c, (R + rc - 1) / rc, 1);
    dim3 g((unsigned)c->n_blockpairs, (R + rc - 1) / rc, sp.nz);
    if (tp == 2) {
        if (rc == 1) launch_sym32<1, 2>(c, g, R, sw, y, sp);
        else if (rc == 2) launch_sym32<2, 2>(c, g, R, sw, y, sp);
        else launch_sym32<4, 2>(c, g, R, sw, y, sp);
    } else {
        if (rc == 1) launch_sym32<1, 1>(c, g, R, sw, y, sp);
        else if (rc == 2) launch_sym32<2, 1>(c, g, R, sw, y, sp);
        else launch_sym32<4, 1>(c, g, R, sw, y, sp);
    }
    cudaError_t e = cudaGetLastError();
    prof_end(c, slot);
    return check_cuda(c, e, "nbody32_sym_kernel");
}

}  // namespace hzb
