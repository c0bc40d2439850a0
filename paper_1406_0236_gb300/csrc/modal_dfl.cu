// Block-diagonal inverse D^{-1} (Sec. 4, Remark after Eq. (precond); Eq. (singleinverse))
// in lean double-float arithmetic on the FP32 pipe: the same three steps as modal.cu
// (azimuthal DFT of every ring, tau^_p = S_|p| y^_p, inverse DFT with the 1/N_F factor
// and tau = alpha sigma + beta tau), for the refinement residual of the mixed solve.
// GB300 runs FP64 at 1/64 of the FP32 rate; a complex multiply-add in double-float
// takes 48 FP32 operations against 4 FP64 fused multiply-adds, so at the two pipes'
// peaks these kernels run about six times faster than the FP64 ones, at about 1e-13
// relative error instead of 1e-16.
//
// Complex values travel as float4 (re.hi, re.lo, im.hi, im.lo): the inputs y and sigma
// and the output tau are FP64 and converted once per element; the mode panels and the
// scattering matrices S_p (split once per build into a cached copy) are double-float.
// Accumulators are renormalised every 16 terms.
#include <algorithm>

#include "hzb_internal.h"
#include "lean_df.cuh"
#include "modal_gemm.cuh"

namespace hzb {

using namespace lean;

static const int DFLM_THREADS = 128;

__global__ void csplit_kernel(size_t n, const double2 *__restrict__ in, float4 *__restrict__ out)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) out[e] = csplit(in[e]);
}

// cos, sin(2 pi m / NF), m < NF, in double-float
__device__ __forceinline__ void dfl_twiddles(int NF, const double2 *__restrict__ tw64, float4 *tw)
{
    for (int m = threadIdx.x; m < NF; m += blockDim.x) tw[m] = csplit(tw64[m]);
}

__device__ __forceinline__ float4 cadd_df(float4 a, float4 b)
{
    const dd x = norm(add({a.x, a.y}, {b.x, b.y})), y = norm(add({a.z, a.w}, {b.z, b.w}));
    return make_float4(x.h, x.l, y.h, y.l);
}
__device__ __forceinline__ float4 cneg_df(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }

// the folded sums of modal.cu (four real double-float multiply-adds per term and two outputs):
// ev += s cos, od += d sin over the M terms of one (mode, right-hand side)
__device__ __forceinline__ void dfl_folded_sums(int M, int NF, int R, int r, int step, const float4 *sv, const float4 *dv,
                                                const float4 *tw, dd (&ev)[2], dd (&od)[2])
{
    ev[0] = ev[1] = od[0] = od[1] = {0.f, 0.f};
    int idx = 0;
    for (int l = 0; l < M; ++l) {
        idx += step;
        if (idx >= NF) idx -= NF;
        const float4 s = sv[l * R + r], d = dv[l * R + r], w = tw[idx];
        const dd c = {w.x, w.y}, sn = {w.z, w.w};
        ev[0] = add(ev[0], mul({s.x, s.y}, c));
        ev[1] = add(ev[1], mul({s.z, s.w}, c));
        od[0] = add(od[0], mul({d.x, d.y}, sn));
        od[1] = add(od[1], mul({d.z, d.w}, sn));
        if ((l & 15) == 15) {
            ev[0] = norm(ev[0]); ev[1] = norm(ev[1]);
            od[0] = norm(od[0]); od[1] = norm(od[1]);
        }
    }
}

// One block per (body of the shape, ring): yh_p = sum_l y(i, l) e^{-2 pi i p l / NF}
__global__ void dfl_dft_forward_kernel(int NG, int NF, int R, int ncols, const long long *__restrict__ body_off,
                                       const double2 *__restrict__ y, const double2 *__restrict__ tw64,
                                       float4 *__restrict__ yh)
{
    extern __shared__ float4 smem_f4[];
    const int M = (NF - 1) / 2;
    float4 *tw = smem_f4;                            // NF
    float4 *y0 = tw + NF;                            // R
    float4 *sv = y0 + R, *dv = sv + (size_t)M * R;   // M x R each
    const int bs = blockIdx.y, i = blockIdx.x;
    const double2 *yr = y + (body_off[bs] + (long long)i * NF) * R;
    dfl_twiddles(NF, tw64, tw);
    for (int e = threadIdx.x; e < (M + 1) * R; e += blockDim.x) {
        const float4 a = csplit(yr[e]);
        if (e < R) {
            y0[e] = a;
        } else {
            const int l = e / R, r = e - l * R;
            const float4 b = csplit(yr[(size_t)(NF - l) * R + r]);
            sv[e - R] = cadd_df(a, b);
            dv[e - R] = cadd_df(a, cneg_df(b));
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < (M + 1) * R; e += blockDim.x) {
        const int p = e / R, r = e - p * R;
        dd ev[2], od[2];
        dfl_folded_sums(M, NF, R, r, p, sv, dv, tw, ev, od);
        const dd cx = add({y0[r].x, y0[r].y}, ev[0]), cy = add({y0[r].z, y0[r].w}, ev[1]);
        const dd px = norm(add(cx, od[1])), py = norm(sub(cy, od[0]));
        const dd mx = norm(sub(cx, od[1])), my = norm(add(cy, od[0]));
        float4 *o = yh + ((size_t)p * NG + i) * ncols + 2 * bs * R + r;
        o[0] = make_float4(px.h, px.l, py.h, py.l);
        o[R] = p ? make_float4(mx.h, mx.l, my.h, my.l) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// tau(i, l) = alpha sigma(i, l) + beta / NF * sum_p tau^_p(i) e^{2 pi i p l / NF}
__global__ void dfl_dft_inverse_kernel(int NG, int NF, int R, int ncols, const long long *__restrict__ body_off,
                                       const float4 *__restrict__ th, const double2 *__restrict__ sigma,
                                       const double2 *__restrict__ tw64, double alpha, double beta,
                                       double2 *__restrict__ out)
{
    extern __shared__ float4 smem_f4[];
    const int M = (NF - 1) / 2;
    float4 *tw = smem_f4;                            // NF
    float4 *t0 = tw + NF;                            // R
    float4 *av = t0 + R, *bv = av + (size_t)M * R;   // M x R each: t_p + t_-p, t_p - t_-p
    const int bs = blockIdx.y, i = blockIdx.x;
    const long long base = (body_off[bs] + (long long)i * NF) * R;
    dfl_twiddles(NF, tw64, tw);
    for (int e = threadIdx.x; e < (M + 1) * R; e += blockDim.x) {
        const int p = e / R, r = e - p * R;
        const float4 *t = th + ((size_t)p * NG + i) * ncols + 2 * bs * R + r;
        const float4 a = t[0];
        if (p == 0) {
            t0[r] = a;
        } else {
            const float4 b = t[R];
            av[e - R] = cadd_df(a, b);
            bv[e - R] = cadd_df(a, cneg_df(b));
        }
    }
    __syncthreads();
    const double sc = beta / NF;
    for (int e = threadIdx.x; e < (M + 1) * R; e += blockDim.x) {
        const int l = e / R, r = e - l * R;
        dd ev[2], od[2];
        dfl_folded_sums(M, NF, R, r, l, av, bv, tw, ev, od);
        const dd cx = add({t0[r].x, t0[r].y}, ev[0]), cy = add({t0[r].z, t0[r].w}, ev[1]);
        auto put = [&](int row, dd x, dd yv) {
            const long long q = base + (long long)row * R + r;
            double2 o = make_double2(value(norm(x)) * sc, value(norm(yv)) * sc);
            if (alpha != 0.0) {
                const double2 s = sigma[q];
                o.x = fma(alpha, s.x, o.x);
                o.y = fma(alpha, s.y, o.y);
            }
            out[q] = o;
        };
        put(l, sub(cx, od[1]), add(cy, od[0]));
        if (l) put(NF - l, add(cx, od[1]), sub(cy, od[0]));
    }
}

// the shape's S_p split into double-float, built on first use after each (re)build
static hzb_status ensure_sdd(hzb_ctx *c, ShapeDev &sd)
{
    if (sd.Sdd_ready) return HZB_OK;
    if (c->capturing) return fail(c, HZB_ESTATE, "double-float scattering matrices not built before capture");
    const size_t nmat = (size_t)(sd.geom.M + 1) * sd.geom.NG * sd.geom.NG;
    if (check_cuda(c, sd.Sdd.ensure(nmat), "alloc double-float S")) return HZB_ENOMEM;
    csplit_kernel<<<(unsigned)((nmat + 255) / 256), 256, 0, c->stream>>>(nmat, sd.S64.ptr, sd.Sdd.ptr);
    c->launches++;
    if (check_cuda(c, cudaGetLastError(), "split S")) return HZB_ECUDA;
    sd.Sdd_ready = true;
    return HZB_OK;
}

// The DFT kernels' dynamic shared memory beyond the default 48 KB: raised once to the
// largest size any call uses (200 KB), never lowered.
static void dfl_dft_smem_limit(size_t bytes)
{
    if (bytes <= 48 * 1024) return;
    cudaFuncSetAttribute(dfl_dft_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(dfl_dft_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

// tau = alpha sigma + beta D^{-1} y with the DFTs and the mode GEMMs in double-float;
// the mode panels live in the FP64 panel buffers (16 bytes per value either way)
hzb_status local_inverse_dfl(hzb_ctx *c, int R, const double2 *y, const double2 *sigma, double alpha, double beta,
                             double2 *tau)
{
    if (c->reduced) return reduced_local(c, R, y, sigma, alpha, beta, tau, false);
    for (ShapeDev *sp : c->shapes) {
        ShapeDev &sd = *sp;
        const int NG = sd.geom.NG, NF = sd.geom.NF, M = sd.geom.M;
        const int ms = (int)sd.bodies.size();
        const int ncols = 2 * ms * R;
        const size_t panel = (size_t)(M + 1) * NG * ncols;
        hzb_status st = ensure_sdd(c, sd);
        if (st) return st;
        if (check_cuda(c, c->yhat64.ensure(panel), "alloc") || check_cuda(c, c->that64.ensure(panel), "alloc"))
            return HZB_ENOMEM;
        float4 *yh = reinterpret_cast<float4 *>(c->yhat64.ptr);
        float4 *th = reinterpret_cast<float4 *>(c->that64.ptr);
        const size_t smem = (size_t)NF * (R + 1) * sizeof(float4);
        if (smem > 200 * 1024) return fail(c, HZB_EINVAL, "n_modes * R too large for the modal apply");
        dfl_dft_smem_limit(smem);
        const long long *doff = sd.body_offs.ptr;
        dfl_dft_forward_kernel<<<dim3(NG, ms), DFLM_THREADS, smem, c->stream>>>(NG, NF, R, ncols, doff, y, sd.tw.ptr,
                                                                                yh);
        modal_gemm<float4, 2, 1>(c->stream, NG, ncols, M + 1, sd.Sdd.ptr, yh, th);
        dfl_dft_inverse_kernel<<<dim3(NG, ms), DFLM_THREADS, smem, c->stream>>>(NG, NF, R, ncols, doff, th, sigma,
                                                                                sd.tw.ptr, alpha, beta, tau);
        c->launches += 3;
        if (check_cuda(c, cudaGetLastError(), "double-float modal apply")) return HZB_ECUDA;
    }
    return HZB_OK;
}

}  // namespace hzb
