// Block-diagonal inverse D^{-1} (Sec. 4, Remark after Eq. (precond); Eq. (singleinverse)):
// for each body, (1) DFT over the azimuth of every ring,
//     y^_p(i) = sum_l y(i, l) e^{-2 pi i p l / N_F},  p = -M..M,
// (2) tau^_p = S_|p| y^_p (S_{-p} = S_p because the modal kernels are even in psi),
// (3) inverse DFT with the 1/N_F factor, and tau = alpha sigma + beta tau.
// Step (2) is a batched complex GEMM per (shape, |p|): the columns stack, for every
// body of that shape, the +p and -p coefficient vectors of all right-hand sides.
// Column layout of a shape's mode-p panel: col = (2 * body_in_shape + sign) * R + r,
// sign 0 for +p and 1 for -p (the -0 columns are zero).
#include <algorithm>

#include "hzb_internal.h"
#include "kernel_math.cuh"
#include "modal_gemm.cuh"
#include "tcgen05.cuh"

namespace hzb {

template <typename T> struct C2;
template <> struct C2<double> { typedef double2 t; };
template <> struct C2<float> { typedef float2 t; };

void launch_modal_gemm_tc(hzb_ctx *c, int n, int nc, int modes, const float2 *A, const float2 *B, float2 *C);

template <typename T> struct alignas(16) Quad { T x, y, z, w; };

// Azimuthal DFTs with the terms l and N_F - l (forward) or +p and -p (inverse) folded: with
// s_l = y_l + y_{N_F - l} and d_l = y_l - y_{N_F - l}, l = 1..M,
//     y^_{+-p} = y_0 + sum_l s_l cos(2 pi p l / N_F) -+ i sum_l d_l sin(2 pi p l / N_F),
// so that four real multiply-adds per (p, l) give two outputs: a quarter of the direct sum's
// (N_F is odd, often prime).  A thread owns PB modes of RB right-hand sides: twiddles and index
// updates are shared by the RB columns, folded values by the PB modes.  The twiddles come from
// the shape's table (make_nodes); computing them in every block took the FP64 pipe longer than
// the sums at small N_F.  258,560 unknowns, R = 16, FP32: forward 197 -> 79 us, inverse
// 188 -> 72 us; 8,200 unknowns, R = 1: 6.4 and 7.0 -> 5.5 and 6.0 us.

// One block per (body of the shape, ring).  y is N x R (FP64); yh is the shape's panel array
// (M+1) x NG x ncols in precision T, which is also the arithmetic precision.
template <typename T, int PB, int RB>
__global__ void __launch_bounds__(128)
dft_forward_kernel(int NG, int NF, int R, int ncols, const long long *__restrict__ body_off,
                   const double2 *__restrict__ y, const double2 *__restrict__ tw64, typename C2<T>::t *__restrict__ yh)
{
    typedef typename C2<T>::t ct;
    extern __shared__ __align__(16) unsigned char dft_smem[];
    const int M = (NF - 1) / 2;
    Quad<T> *sd = (Quad<T> *)dft_smem;               // M x R: s, d
    ct *y0 = (ct *)(sd + (size_t)M * R);             // R
    ct *tw = y0 + R;                                 // NF: cos, sin(2 pi m / NF)
    const int bs = blockIdx.y, i = blockIdx.x;
    const double2 *yr = y + (body_off[bs] + (long long)i * NF) * R;
    for (int m = threadIdx.x; m < NF; m += blockDim.x) {
        const double2 v = tw64[m];
        tw[m].x = (T)v.x;
        tw[m].y = (T)v.y;
    }
    for (int e = threadIdx.x; e < (M + 1) * R; e += blockDim.x) {
        const double2 a = yr[e];
        if (e < R) {
            y0[e].x = (T)a.x;
            y0[e].y = (T)a.y;
        } else {
            const int l = e / R, r = e - l * R;
            const double2 b = yr[(size_t)(NF - l) * R + r];
            const T ax = (T)a.x, ay = (T)a.y, bx = (T)b.x, by = (T)b.y;
            sd[e - R] = {ax + bx, ay + by, ax - bx, ay - by};
        }
    }
    __syncthreads();
    const int nrb = (R + RB - 1) / RB, items = ((M + PB) / PB) * nrb;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const int p0 = (it / nrb) * PB, r0 = it % nrb;
        Quad<T> acc[PB][RB];                         // sum s cos, sum d sin
        int idx[PB];
#pragma unroll
        for (int q = 0; q < PB; ++q) {
            idx[q] = 0;
#pragma unroll
            for (int u = 0; u < RB; ++u) acc[q][u] = {(T)0, (T)0, (T)0, (T)0};
        }
#pragma unroll 2
        for (int l = 0; l < M; ++l) {
            Quad<T> v[RB];
#pragma unroll
            for (int u = 0; u < RB; ++u) v[u] = sd[l * R + min(r0 + nrb * u, R - 1)];
#pragma unroll
            for (int q = 0; q < PB; ++q) {
                idx[q] += p0 + q;
                if (idx[q] >= NF) idx[q] -= NF;
                const ct w = tw[idx[q]];
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    acc[q][u].x = fma(v[u].x, w.x, acc[q][u].x);
                    acc[q][u].y = fma(v[u].y, w.x, acc[q][u].y);
                    acc[q][u].z = fma(v[u].z, w.y, acc[q][u].z);
                    acc[q][u].w = fma(v[u].w, w.y, acc[q][u].w);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < PB; ++q) {
            const int p = p0 + q;
            if (p > M) break;
            ct *o = yh + ((size_t)p * NG + i) * ncols + 2 * bs * R;
#pragma unroll
            for (int u = 0; u < RB; ++u) {
                const int r = r0 + nrb * u;
                if (r >= R) break;
                const Quad<T> A = acc[q][u];
                const ct z = y0[r];
                const T cx = z.x + A.x, cy = z.y + A.y;
                ct plus, minus;
                plus.x = cx + A.w; plus.y = cy - A.z;
                minus.x = p ? cx - A.w : (T)0; minus.y = p ? cy + A.z : (T)0;     // the -0 columns are zero
                o[r] = plus;
                o[R + r] = minus;
            }
        }
    }
}

// tau(i, l) = alpha sigma(i, l) + beta / NF * sum_p tau^_p(i) e^{2 pi i p l / NF}
template <typename T, int PB, int RB>
__global__ void __launch_bounds__(128)
dft_inverse_kernel(int NG, int NF, int R, int ncols, const long long *__restrict__ body_off,
                   const typename C2<T>::t *__restrict__ th, const double2 *__restrict__ sigma,
                   const double2 *__restrict__ tw64, double alpha, double beta, double2 *__restrict__ out)
{
    typedef typename C2<T>::t ct;
    extern __shared__ __align__(16) unsigned char dft_smem[];
    const int M = (NF - 1) / 2;
    Quad<T> *ab = (Quad<T> *)dft_smem;               // M x R: t_p + t_-p, t_p - t_-p
    ct *t0 = (ct *)(ab + (size_t)M * R);             // R
    ct *tw = t0 + R;                                 // NF: cos, sin(2 pi m / NF)
    const int bs = blockIdx.y, i = blockIdx.x;
    const long long base = (body_off[bs] + (long long)i * NF) * R;
    for (int m = threadIdx.x; m < NF; m += blockDim.x) {
        const double2 v = tw64[m];
        tw[m].x = (T)v.x;
        tw[m].y = (T)v.y;
    }
    for (int e = threadIdx.x; e < (M + 1) * R; e += blockDim.x) {
        const int p = e / R, r = e - p * R;
        const ct *t = th + ((size_t)p * NG + i) * ncols + 2 * bs * R + r;
        const ct a = t[0];
        if (p == 0) {
            t0[r] = a;
        } else {
            const ct b = t[R];
            ab[e - R] = {a.x + b.x, a.y + b.y, a.x - b.x, a.y - b.y};
        }
    }
    __syncthreads();
    const double sc = beta / NF;
    const int nrb = (R + RB - 1) / RB, items = ((M + PB) / PB) * nrb;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const int l0 = (it / nrb) * PB, r0 = it % nrb;
        Quad<T> acc[PB][RB];
        int idx[PB];
#pragma unroll
        for (int q = 0; q < PB; ++q) {
            idx[q] = 0;
#pragma unroll
            for (int u = 0; u < RB; ++u) acc[q][u] = {(T)0, (T)0, (T)0, (T)0};
        }
#pragma unroll 2
        for (int p = 0; p < M; ++p) {
            Quad<T> v[RB];
#pragma unroll
            for (int u = 0; u < RB; ++u) v[u] = ab[p * R + min(r0 + nrb * u, R - 1)];
#pragma unroll
            for (int q = 0; q < PB; ++q) {
                idx[q] += l0 + q;
                if (idx[q] >= NF) idx[q] -= NF;
                const ct w = tw[idx[q]];
#pragma unroll
                for (int u = 0; u < RB; ++u) {
                    acc[q][u].x = fma(v[u].x, w.x, acc[q][u].x);
                    acc[q][u].y = fma(v[u].y, w.x, acc[q][u].y);
                    acc[q][u].z = fma(v[u].z, w.y, acc[q][u].z);
                    acc[q][u].w = fma(v[u].w, w.y, acc[q][u].w);
                }
            }
        }
        auto put = [&](int l, int r, T x, T yv) {
            const long long e = base + (long long)l * R + r;
            double2 o = make_double2((double)x * sc, (double)yv * sc);
            if (alpha != 0.0) {
                const double2 s = sigma[e];
                o.x = fma(alpha, s.x, o.x);
                o.y = fma(alpha, s.y, o.y);
            }
            out[e] = o;
        };
#pragma unroll
        for (int q = 0; q < PB; ++q) {
            const int l = l0 + q;
            if (l > M) break;
#pragma unroll
            for (int u = 0; u < RB; ++u) {
                const int r = r0 + nrb * u;
                if (r >= R) break;
                const Quad<T> A = acc[q][u];
                const ct z = t0[r];
                const T cx = z.x + A.x, cy = z.y + A.y;
                put(l, r, cx - A.w, cy + A.z);
                if (l) put(NF - l, r, cx + A.w, cy - A.z);
            }
        }
    }
}

// One thread per (two or four modes, four right-hand sides), fewer where the batch is smaller.  The
// dynamic shared memory limit is raised once beyond the default 48 KB, to the largest size any
// call uses, and never lowered, so that calls with different sizes (and both D^{-1} entry
// points) cannot invalidate each other's launches.
template <typename T>
static size_t dft_smem(int NF, int R)
{
    return (size_t)NF * (R + 1) * sizeof(typename C2<T>::t);
}

template <typename K>
static void dft_limit(K kern, size_t bytes)
{
    if (bytes > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

// Four modes to a thread, where that leaves blocks of 48 threads and 16,384 of them in all: the
// reads from shared memory bound these kernels (258,560 unknowns, FP32: R = 16, 52 threads, 96 -> 79
// and 85 -> 72 us; R = 8, 26 threads, 3 % slower; 8,200 unknowns: R = 64, 96 threads, whole D^{-1}
// 66 -> 58, R = 16, 24 threads, 29 -> 38).
static bool dft_wide(int M, int R, long long blocks)
{
    const int threads = (M + 4) / 4 * ((R + 3) / 4);
    return R >= 4 && threads >= 48 && blocks * threads >= 16384;
}

static int dft_threads(int items) { return std::min(128, std::max(32, (items + 31) / 32 * 32)); }

template <typename T>
static void dft_forward(cudaStream_t st, const ShapeDev &sd, int ms, int R, const long long *off, const double2 *y,
                        typename C2<T>::t *yh)
{
    const int NG = sd.geom.NG, NF = sd.geom.NF, M = sd.geom.M, ncols = 2 * ms * R;
    const size_t smem = dft_smem<T>(NF, R);
    auto launch = [&](auto kern, int pb, int rb) {
        dft_limit(kern, smem);
        kern<<<dim3(NG, ms), dft_threads((M + pb) / pb * ((R + rb - 1) / rb)), smem, st>>>(NG, NF, R, ncols, off, y,
                                                                                     sd.tw.ptr, yh);
    };
    if (dft_wide(M, R, NG * ms)) launch(dft_forward_kernel<T, 4, 4>, 4, 4);
    else if (R >= 4) launch(dft_forward_kernel<T, 2, 4>, 2, 4);
    else if (R >= 2) launch(dft_forward_kernel<T, 1, 2>, 1, 2);
    else launch(dft_forward_kernel<T, 1, 1>, 1, 1);
}

template <typename T>
static void dft_inverse(cudaStream_t st, const ShapeDev &sd, int ms, int R, const long long *off,
                        const typename C2<T>::t *th, const double2 *sigma, double alpha, double beta, double2 *out)
{
    const int NG = sd.geom.NG, NF = sd.geom.NF, M = sd.geom.M, ncols = 2 * ms * R;
    const size_t smem = dft_smem<T>(NF, R);
    auto launch = [&](auto kern, int pb, int rb) {
        dft_limit(kern, smem);
        kern<<<dim3(NG, ms), dft_threads((M + pb) / pb * ((R + rb - 1) / rb)), smem, st>>>(
            NG, NF, R, ncols, off, th, sigma, sd.tw.ptr, alpha, beta, out);
    };
    if (dft_wide(M, R, NG * ms)) launch(dft_inverse_kernel<T, 4, 4>, 4, 4);
    else if (R >= 4) launch(dft_inverse_kernel<T, 2, 4>, 2, 4);
    else if (R >= 2) launch(dft_inverse_kernel<T, 1, 2>, 1, 2);
    else launch(dft_inverse_kernel<T, 1, 1>, 1, 1);
}

// Below this the two launches, the embedding pass and the few blocks of the TMA form cost more
// than the tensor cores save.  Whole D^{-1}, CUDA cores against TMA (us): N_G = 100, 21 modes,
// 32 / 64 / 256 columns (7 / 13 / 54e6) 27 / 29 / 66 against 36 / 40 / 73; N_G = 144: 31 / 34 / 82
// against 38 / 44 / 78 (14 / 28 / 111e6); N_G = 224, 31 modes: 44 / 64 against 48 / 58
// (50 / 100e6); N_G = 320, 51 modes, 32 columns (167e6): 94 against 88.
static const double MODAL_TMA_MIN = 6e7;

template <typename T>
static hzb_status local_inverse_t(hzb_ctx *c, int R, const double2 *y, const double2 *sigma, double alpha,
                                  double beta, double2 *tau)
{
    typedef typename C2<T>::t ct;
    if (c->reduced) return reduced_local(c, R, y, sigma, alpha, beta, tau, sizeof(T) == 4);
    for (ShapeDev *sp : c->shapes) {
        ShapeDev &sd = *sp;
        const int NG = sd.geom.NG, NF = sd.geom.NF, M = sd.geom.M;
        const int ms = (int)sd.bodies.size();
        const int ncols = 2 * ms * R;
        const size_t panel = (size_t)(M + 1) * NG * ncols;
        ct *yh, *th;
        const ct *S;
        if (sizeof(T) == 8) {
            if (check_cuda(c, c->yhat64.ensure(panel), "alloc") || check_cuda(c, c->that64.ensure(panel), "alloc"))
                return HZB_ENOMEM;
            yh = (ct *)c->yhat64.ptr;
            th = (ct *)c->that64.ptr;
            S = (const ct *)sd.S64.ptr;
        } else {
            if (check_cuda(c, c->yhat32.ensure(panel), "alloc") || check_cuda(c, c->that32.ensure(panel), "alloc"))
                return HZB_ENOMEM;
            yh = (ct *)c->yhat32.ptr;
            th = (ct *)c->that32.ptr;
            S = (const ct *)sd.S32.ptr;
        }
        const long long *doff = sd.body_offs.ptr;        // first node of each body of the shape
        if (dft_smem<T>(NF, R) > 200 * 1024) return fail(c, HZB_EINVAL, "n_modes * R too large for the modal apply");
        dft_forward<T>(c->stream, sd, ms, R, doff, y, yh);
        // FP32 path: tcgen05 fed by TMA (modal_tma.cu) from 32 columns and MODAL_TMA_MIN complex
        // multiply-adds on, or as chosen; mma.sync TF32 x 3 on request
        const bool f32 = sizeof(T) == 4;
        const double macs = (double)(M + 1) * NG * NG * ncols;
        if (f32 && (c->modal_engine == 2 || (c->modal_engine < 0 && ncols >= 32 && macs >= MODAL_TMA_MIN))) {
            hzb_status st = modal_gemm_tma(c, sd, ncols, (const float2 *)yh, (float2 *)th);
            if (st) return st;
        } else if (f32 && c->modal_engine == 1)
            launch_modal_gemm_tc(c, NG, ncols, M + 1, (const float2 *)S, (const float2 *)yh, (float2 *)th);
        else
            modal_gemm<ct, 2, 1>(c->stream, NG, ncols, M + 1, S, yh, th);
        dft_inverse<T>(c->stream, sd, ms, R, doff, th, sigma, alpha, beta, tau);
        c->launches += 3;
        if (check_cuda(c, cudaGetLastError(), "modal apply")) return HZB_ECUDA;
    }
    return HZB_OK;
}

hzb_status local_inverse64(hzb_ctx *c, int R, const double2 *y, const double2 *sigma, double alpha, double beta,
                           double2 *tau)
{
    return local_inverse_t<double>(c, R, y, sigma, alpha, beta, tau);
}

hzb_status local_inverse32(hzb_ctx *c, int R, const double2 *y, const double2 *sigma, double alpha, double beta,
                           double2 *tau)
{
    return local_inverse_t<float>(c, R, y, sigma, alpha, beta, tau);
}

}  // namespace hzb

namespace hzb {

// The FP64 D^{-1} apply with caller-provided scratch: yh and th each hold at least
// (M+1) x N_G x (2 m_s R) complex values for every shape (shapes run one after the
// other on the stream, reusing them).  Launches the same kernels as local_inverse64
// and allocates nothing.
hzb_status local_inverse64_scratch(hzb_ctx *c, int R, const double2 *y, const double2 *sigma, double alpha,
                                   double beta, double2 *tau, double2 *yh, double2 *th)
{
    for (ShapeDev *sp : c->shapes) {
        ShapeDev &sd = *sp;
        const int NG = sd.geom.NG, M = sd.geom.M, ms = (int)sd.bodies.size();
        const long long *doff = sd.body_offs.ptr;
        if (dft_smem<double>(sd.geom.NF, R) > 200 * 1024)
            return fail(c, HZB_EINVAL, "n_modes * R too large for the modal apply");
        dft_forward<double>(c->stream, sd, ms, R, doff, y, yh);
        modal_gemm<double2, 2, 1>(c->stream, NG, 2 * ms * R, M + 1, sd.S64.ptr, yh, th);
        dft_inverse<double>(c->stream, sd, ms, R, doff, th, sigma, alpha, beta, tau);
        c->launches += 3;
        if (check_cuda(c, cudaGetLastError(), "modal apply")) return HZB_ECUDA;
    }
    return HZB_OK;
}

// Y = A_pp^{-1} X for a single body of the shape placed at offset 0 (X, Y: n x R,
// node-major), FP64: the same three kernels as local_inverse64.
hzb_status shape_inverse64(hzb_ctx *c, ShapeDev &sd, int R, const double2 *X, double2 *Y)
{
    const int NG = sd.geom.NG, NF = sd.geom.NF, M = sd.geom.M;
    const int ncols = 2 * R;
    const size_t panel = (size_t)(M + 1) * NG * ncols;
    if (check_cuda(c, c->yhat64.ensure(panel), "alloc") || check_cuda(c, c->that64.ensure(panel), "alloc") ||
        check_cuda(c, c->zero_off.ensure(1), "alloc"))
        return HZB_ENOMEM;
    if (check_cuda(c, cudaMemsetAsync(c->zero_off.ptr, 0, sizeof(long long), c->stream), "memset")) return HZB_ECUDA;
    if (dft_smem<double>(NF, R) > 200 * 1024) return fail(c, HZB_EINVAL, "n_modes * R too large for the modal apply");
    dft_forward<double>(c->stream, sd, 1, R, c->zero_off.ptr, X, c->yhat64.ptr);
    modal_gemm<double2, 2, 1>(c->stream, NG, ncols, M + 1, sd.S64.ptr, c->yhat64.ptr, c->that64.ptr);
    dft_inverse<double>(c->stream, sd, 1, R, c->zero_off.ptr, c->that64.ptr, nullptr, 0.0, 1.0, Y);
    c->launches += 3;
    return check_cuda(c, cudaGetLastError(), "shape inverse");
}

// Largest per-shape panel (M+1) x N_G x (2 m_s R) of the context, in complex values.
size_t modal_panel_elems(const hzb_ctx *c, int R)
{
    size_t mx = 0;
    for (const ShapeDev *sp : c->shapes)
        mx = std::max(mx, (size_t)(sp->geom.M + 1) * sp->geom.NG * (2 * sp->bodies.size() * (size_t)R));
    return mx;
}

}  // namespace hzb

namespace hzb {

// ---------------------------------------------------------------- tensor-core modal GEMM
// FP32 path, many columns: C = A B for complex A (n x n) and B (n x nc) through the
// real embedding  [Cr; Ci] = [[Ar, -Ai], [Ai, Ar]] [Br; Bi]  (a 2n x 2n x nc real GEMM)
// on the tensor cores in TF32 with a three-term split, x = hi + lo with hi, lo TF32:
// A B ~ Ahi Bhi + Ahi Blo + Alo Bhi, FP32 accumulation (about FP32 accuracy).
// mma.sync m16n8k8; 64 x 64 output tile per CTA, 4 warps of 32 x 32, K step 32.

__device__ __forceinline__ uint32_t to_tf32(float x)       // = cvt.rna.tf32.f32 for finite x
{
    return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u;
}

__device__ __forceinline__ void mma_tf32(float *d, const uint32_t *a, const uint32_t *b)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__global__ void __launch_bounds__(128)
modal_gemm_tc_kernel(int n, int nc, const float2 *__restrict__ A, const float2 *__restrict__ B, float2 *__restrict__ C)
{
    __shared__ float As[64][33];
    __shared__ float Bs[32][72];
    const int p = blockIdx.z;
    const float2 *Ap = A + (size_t)p * n * n;
    const float2 *Bp = B + (size_t)p * n * nc;
    float2 *Cp = C + (size_t)p * n * nc;
    const int n2 = 2 * n;
    const int row0 = blockIdx.y * 64, col0 = blockIdx.x * 64;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 1, wn = warp & 1;
    const int g = lane >> 2, t = lane & 3;
    float acc[2][4][4];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
    for (int k0 = 0; k0 < n2; k0 += 32) {
        for (int e = tid; e < 64 * 32; e += 128) {
            const int r = e >> 5, kk = e & 31;
            const int R = row0 + r, K = k0 + kk;
            float v = 0.f;
            if (R < n2 && K < n2) {
                const float2 a = Ap[(size_t)(R < n ? R : R - n) * n + (K < n ? K : K - n)];
                v = (R < n) ? (K < n ? a.x : -a.y) : (K < n ? a.y : a.x);
            }
            As[r][kk] = v;
        }
        for (int e = tid; e < 32 * 64; e += 128) {
            const int kk = e >> 6, c = e & 63;
            const int K = k0 + kk, col = col0 + c;
            float v = 0.f;
            if (K < n2 && col < nc) {
                const float2 b = Bp[(size_t)(K < n ? K : K - n) * nc + col];
                v = (K < n) ? b.x : b.y;
            }
            Bs[kk][c] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 32; kk += 8) {
            uint32_t ah[2][4], al[2][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const int r = wm * 32 + mt * 16 + g;
                const float v[4] = {As[r][kk + t], As[r + 8][kk + t], As[r][kk + t + 4], As[r + 8][kk + t + 4]};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    ah[mt][q] = to_tf32(v[q]);
                    al[mt][q] = to_tf32(v[q] - __uint_as_float(ah[mt][q]));
                }
            }
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int c = wn * 32 + nt * 8 + g;
                const float v0 = Bs[kk + t][c], v1 = Bs[kk + t + 4][c];
                const uint32_t bh[2] = {t5_tf32(v0), t5_tf32(v1)};       // (keeps a NaN of the panel)
                const uint32_t bl[2] = {t5_tf32(v0 - __uint_as_float(bh[0])), t5_tf32(v1 - __uint_as_float(bh[1]))};
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    mma_tf32(acc[mt][nt], al[mt], bh);
                    mma_tf32(acc[mt][nt], ah[mt], bl);
                    mma_tf32(acc[mt][nt], ah[mt], bh);
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int R = row0 + wm * 32 + mt * 16 + g + 8 * h;
                const int col = col0 + wn * 32 + nt * 8 + 2 * t;
                if (R >= n2) continue;
                float *base = (R < n) ? &Cp[(size_t)R * nc].x : &Cp[(size_t)(R - n) * nc].y;
                if (col < nc) base[2 * col] = acc[mt][nt][2 * h];
                if (col + 1 < nc) base[2 * (col + 1)] = acc[mt][nt][2 * h + 1];
            }
}

void launch_modal_gemm_tc(hzb_ctx *c, int n, int nc, int modes, const float2 *A, const float2 *B, float2 *C)
{
    dim3 grid((nc + 63) / 64, (2 * n + 63) / 64, modes);
    modal_gemm_tc_kernel<<<grid, 128, 0, c->stream>>>(n, nc, A, B, C);
}

}  // namespace hzb
