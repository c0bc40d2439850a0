// Inter-body sum y = B sigma (Sec. 3.3, Eq. (nystromnaive)) for many right-hand
// sides, with the contraction over sources on the tensor cores.
//
// For a tile of 32 sources and the 32 targets of a warp, the pair kernels
// G(t, s) = e^{ikr}[n_s.d / r^3 - i (k n_s.d / r^2 + eta / r)] (FP32, phase reduced to a
// fraction of a turn as in nbody32_kernel) are generated by the lanes directly in the
// register layout of the B operand of mma.m16n8k8 (each lane computes the two pairs its
// fragment holds), and the weighted densities sigma'(r, s) = w_s sigma_s,r / (4 pi) of
// RC right-hand sides form the A operand (from shared memory).  With
//     Y^T = Sigma'^T G^T:   Yr = Sr Gr - Si Gi,   Yi = Si Gr + Sr Gi,
// each of the four real products runs in TF32 with a three-term hi/lo split
// (x = hi + lo: A B ~ Ahi Bhi + Ahi Blo + Alo Bhi) and FP32 accumulation inside each
// 32-source tile; the tiles' sums are added with rounded FP32 adds, which keeps FP32
// accuracy over millions of sources.  CTA = 4 warps = 128 targets of one TargetBlock (4 CTAs per block);
// grid y = chunks of RC right-hand sides; grid z = source chunks (as nbody32_kernel).
#include <algorithm>

#include "hzb_internal.h"
#include "kernel_math.cuh"
#include "tcgen05.cuh"

namespace hzb {

static const int TC_TBLOCK = 512;
static const int TC_CTA_TARGETS = 128;
static const int TC_S = 32;               // sources per tile

// TF32 operand (round to nearest, ties away, 10 mantissa bits) by two integer operations
// on the bit pattern: equal to cvt.rna.tf32.f32 for finite x, and faster than it (a NaN is lost)
__device__ __forceinline__ uint32_t tf32_of(float x) { return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u; }

__device__ __forceinline__ void mma_m16n8k8(float *d, const uint32_t *a, const uint32_t *b)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// d += (ahi + alo)(bhi + blo) without the lo*lo term
__device__ __forceinline__ void mma3(float *d, const uint32_t *ahi, const uint32_t *alo, const uint32_t *bhi,
                                     const uint32_t *blo)
{
    mma_m16n8k8(d, alo, bhi);
    mma_m16n8k8(d, ahi, blo);
    mma_m16n8k8(d, ahi, bhi);
}

__device__ __forceinline__ void pair_kernel32(float tx, float ty, float tz, float4 a, float2 b, float k, float eta,
                                              float kt, float &gre, float &gim)
{
    const float dx = tx - a.x, dy = ty - a.y, dz = tz - a.z;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float ir = rsqrtf(r2);
    const float nd = fmaf(a.w, dx, fmaf(b.x, dy, b.y * dz));
    const float ndir2 = nd * (ir * ir);
    const float A = ndir2 * ir;
    const float B = fmaf(k, ndir2, eta * ir);
    float turns = (r2 * ir) * kt;
    turns -= rintf(turns);
    float s, c;
    __sincosf(turns * 6.283185307179586f, &s, &c);
    gre = fmaf(c, A, s * B);
    gim = fmaf(s, A, -c * B);
}

template <int MT>
__global__ void __launch_bounds__(128)
nbody_tc_kernel(const TargetBlock *__restrict__ blocks, int N, int R, int chunk, const float4 *__restrict__ pos,
                const float4 *__restrict__ nrm, const float2 *__restrict__ sw, float k, float eta, float kt,
                float2 *__restrict__ ypart, double2 *__restrict__ y, size_t split_stride)
{
    constexpr int RC = 16 * MT;
    constexpr int LD = TC_S + 4;                      // padded row: conflict-free fragment loads
    __shared__ float4 s_a[TC_S];                      // x, y, z, nx
    __shared__ float2 s_b[TC_S];                      // ny, nz
    __shared__ uint32_t s_rh[RC * LD], s_rl[RC * LD], s_ih[RC * LD], s_il[RC * LD];
    const TargetBlock tb = blocks[blockIdx.x >> 2];
    const int sub = blockIdx.x & 3;
    if (sub * TC_CTA_TARGETS >= tb.count) return;              // whole CTA past the block's end
    const int r0 = blockIdx.y * RC;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int wbase = sub * TC_CTA_TARGETS + warp * 32;      // first target (in the block) of this warp
    float tx[4], ty[4], tz[4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int q = wbase + nt * 8 + g;
        float4 p = (q < tb.count) ? pos[tb.start + q] : make_float4(1e18f, 1e18f, 1e18f, 0.f);
        tx[nt] = p.x; ty[nt] = p.y; tz[nt] = p.z;
    }
    // acc: running sums (IEEE FP32 adds); tac: the current tile's tensor-core sums.
    // The tensor cores' internal FP32 accumulation is not rounded to nearest, so a
    // chain of tens of thousands of mma accumulations drifts; each tile starts from 0.
    float acc[MT][4][2][4], tac[MT][4][2][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[m][nt][c][q] = 0.f;
    const bool active = wbase < tb.count;                       // warp has targets
    const int c0 = blockIdx.z * chunk, c1 = min(N, c0 + chunk);
    for (int range = 0; range < 2; ++range) {
        const int lo = range ? max(c0, tb.excl_hi) : c0;
        const int hi = range ? c1 : min(c1, tb.excl_lo);
        for (int j0 = lo; j0 < hi; j0 += TC_S) {
            const int cnt = min(TC_S, hi - j0);
            __syncthreads();
            if (tid < TC_S) {
                if (tid < cnt) {
                    const float4 p = pos[j0 + tid];
                    const float4 n = nrm[j0 + tid];
                    s_a[tid] = make_float4(p.x, p.y, p.z, n.x);
                    s_b[tid] = make_float2(n.y, n.z);
                } else {
                    s_a[tid] = make_float4(-1e18f, -1e18f, -1e18f, 0.f);     // far away: G ~ 0, finite
                    s_b[tid] = make_float2(0.f, 0.f);
                }
            }
            for (int e = tid; e < TC_S * RC; e += 128) {
                const int s = e / RC, r = e % RC;
                float sr = 0.f, si = 0.f;
                if (s < cnt && r0 + r < R) {
                    const float2 v = sw[(size_t)(j0 + s) * R + r0 + r];
                    sr = v.x;
                    si = v.y;
                }
                const uint32_t rh = t5_tf32(sr), ih = t5_tf32(si);       // (keeps a NaN)
                s_rh[r * LD + s] = rh;
                s_rl[r * LD + s] = t5_tf32(sr - __uint_as_float(rh));
                s_ih[r * LD + s] = ih;
                s_il[r * LD + s] = t5_tf32(si - __uint_as_float(ih));
            }
            __syncthreads();
            if (!active) continue;
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int c = 0; c < 2; ++c)
#pragma unroll
                        for (int q = 0; q < 4; ++q) tac[m][nt][c][q] = 0.f;
#pragma unroll
            for (int ks = 0; ks < TC_S / 8; ++ks) {
                // A fragments (rows: right-hand sides, cols: sources) for every m-tile
                uint32_t arh[MT][4], arl[MT][4], aih[MT][4], ail[MT][4], nih[MT][4], nil[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const int rr = m * 16 + g, cc = ks * 8 + t;
                    const int idx[4] = {rr * LD + cc, (rr + 8) * LD + cc, rr * LD + cc + 4, (rr + 8) * LD + cc + 4};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        arh[m][q] = s_rh[idx[q]];
                        arl[m][q] = s_rl[idx[q]];
                        aih[m][q] = s_ih[idx[q]];
                        ail[m][q] = s_il[idx[q]];
                        nih[m][q] = aih[m][q] ^ 0x80000000u;      // -Si
                        nil[m][q] = ail[m][q] ^ 0x80000000u;
                    }
                }
                const int s0 = ks * 8 + t;
                const float4 A0 = s_a[s0], A1 = s_a[s0 + 4];
                const float2 B0 = s_b[s0], B1 = s_b[s0 + 4];
#pragma unroll
                for (int nt = 0; nt < 4; ++nt) {
                    // B fragment of G^T: (source s0, target g) and (source s0 + 4, target g)
                    float g0r, g0i, g1r, g1i;
                    pair_kernel32(tx[nt], ty[nt], tz[nt], A0, B0, k, eta, kt, g0r, g0i);
                    pair_kernel32(tx[nt], ty[nt], tz[nt], A1, B1, k, eta, kt, g1r, g1i);
                    uint32_t brh[2] = {tf32_of(g0r), tf32_of(g1r)};
                    uint32_t brl[2] = {tf32_of(g0r - __uint_as_float(brh[0])), tf32_of(g1r - __uint_as_float(brh[1]))};
                    uint32_t bih[2] = {tf32_of(g0i), tf32_of(g1i)};
                    uint32_t bil[2] = {tf32_of(g0i - __uint_as_float(bih[0])), tf32_of(g1i - __uint_as_float(bih[1]))};
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        mma3(tac[m][nt][0], arh[m], arl[m], brh, brl);      // Yr += Sr Gr
                        mma3(tac[m][nt][0], nih[m], nil[m], bih, bil);      // Yr -= Si Gi
                        mma3(tac[m][nt][1], aih[m], ail[m], brh, brl);      // Yi += Si Gr
                        mma3(tac[m][nt][1], arh[m], arl[m], bih, bil);      // Yi += Sr Gi
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int c = 0; c < 2; ++c)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[m][nt][c][q] += tac[m][nt][c][q];
        }
    }
    // C fragment of Y^T: rows = right-hand sides (g, g + 8), cols = targets (2t, 2t + 1)
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + m * 16 + g + ((q & 2) ? 8 : 0);
                const int tq = wbase + nt * 8 + 2 * t + (q & 1);
                if (r < R && tq < tb.count) {
                    const size_t e = (size_t)(tb.start + tq) * R + r;
                    const float2 v = make_float2(acc[m][nt][0][q], acc[m][nt][1][q]);
                    if (ypart) ypart[blockIdx.z * split_stride + e] = v;
                    else y[e] = make_double2((double)v.x, (double)v.y);
                }
            }
}

hzb_status interbody_tc(hzb_ctx *c, int R, const double2 *sigma, double2 *y, int nsplit)
{
    if (!c->nodes_ready) return fail(c, HZB_ESTATE, "nodes not built");
    const int N = (int)c->N;
    const int RC = 16;                    // one m16 tile of right-hand sides per CTA (MT = 1)
    int chunk = (N + nsplit - 1) / nsplit;
    chunk = ((chunk + TC_S - 1) / TC_S) * TC_S;
    nsplit = (N + chunk - 1) / chunk;
    const size_t n = (size_t)N * R;
    float2 *part = nullptr;
    if (nsplit > 1) {
        if (check_cuda(c, c->nb_part32.ensure(n * nsplit), "alloc partial sums")) return HZB_ENOMEM;
        part = c->nb_part32.ptr;
    }
    c->interbody_calls++;
    c->launches += (nsplit > 1) ? 2 : 1;
    const int slot = prof_begin(c, 1);
    const float2 *sw = weighted_sigma32(c, R, sigma);
    if (!sw) return HZB_ENOMEM;
    const int nb = (c->tune_limit_blocks > 0) ? std::min(c->tune_limit_blocks, c->n_tblocks) : c->n_tblocks;
    dim3 grid(nb * (TC_TBLOCK / TC_CTA_TARGETS), (R + RC - 1) / RC, nsplit);
    const float k = (float)c->k, eta = (float)c->eta, kt = (float)(c->k / (2.0 * M_PI));
    nbody_tc_kernel<1><<<grid, 128, 0, c->stream>>>(c->tblocks.ptr, N, R, chunk, c->pos32.ptr, c->nrm32.ptr, sw, k,
                                                    eta, kt, part, y, n);
    if (nsplit > 1) split_reduce_f2(c, n, nsplit, part, y);
    cudaError_t e = cudaGetLastError();
    prof_end(c, slot);
    return check_cuda(c, e, "nbody_tc_kernel");
}

}  // namespace hzb
