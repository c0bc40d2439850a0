// One pair of nodes in lean double-float: geometry, phase and kernel value of the inter-body sum
// (the formulas and the arithmetic are described in nbody_dfl.cu).  Translation units that include
// this are compiled with -fmad=false.
#pragma once

#include "hzb_internal.h"
#include "lean_df.cuh"

namespace hzb {

using namespace lean;

static const int DFL_S = 32;           // sources per tile
static const int DFL_TAB = 1024;       // table angles 2 pi m / 1024

struct DflConst {
    dd kappa;                          // 2 pi (0 when k = 0)
    float eta_m, mb;                   // eta' rounded onto the grid of mb, plus mb; mb = 1.5 * 2^E for kr X + eta'
    float eta_r;                       // eta' minus its grid value (its low part included)
    float kbound;                      // 2 pi + |eta'|, rounded up
    int no_phase;                      // k = 0
};

// a value of magnitude below 2^(e + 1) with e the exponent of `bound` stays inside the
// binade of this 1.5 * 2^(e + 2) when added to it
__device__ __forceinline__ float dfl_magic_of(float bound)
{
    return __int_as_float((__float_as_int(bound) & 0x7f800000) + 0x01400000);
}

// ulp of a number 1.5 * 2^E
__device__ __forceinline__ float dfl_ulp_of(float m)
{
    return __int_as_float((__float_as_int(m) & 0x7f800000) - (23 << 23));
}

// e^{2 pi i theta} for theta (turns) with |theta| < 2^21; high parts on the grid of ulp(3)
__device__ __forceinline__ void dfl_cis(dd theta, const float4 *__restrict__ tab, dd &cs, dd &sn)
{
    const float MAGIC = 12582912.0f;                      // 1.5 * 2^23: adding it rounds to an integer
    const float n0 = (theta.h + MAGIC) - MAGIC;
    const float f = theta.h - n0;                         // exact, |f| <= 1/2
    const float tm = fmaf(f, (float)DFL_TAB, MAGIC);
    const float mf = tm - MAGIC;                          // nearest table index, as a float
    const int idx = __float_as_int(tm) & (DFL_TAB - 1);   // its low bits are the integer
    const float g = fmaf(mf, -1.0f / DFL_TAB, f);         // exact: |g| <= 1/2048 turns
    // g is zero or a multiple of ulp(theta.h): the fast two-sum is exact
    const float gs = g + theta.l;
    const dd twopi = {6.28318548f, -1.74845553e-7f};
    const dd del = mul({gs, theta.l - (gs - g)}, twopi);  // remainder in radians, |delta| <= pi/1024
    const float q = del.h * del.h;
    const float qe = fmaf(del.h + del.h, del.l, fmaf(del.h, del.h, -q));   // delta^2 = q + qe
    const dd cm = {-0.5f * q, fmaf(q, q * (1.0f / 24.0f), -0.5f * qe)};     // cos(delta) - 1
    const dd sd = {del.h, fmaf(del.h * q, fmaf(q, 1.0f / 120.0f, -1.0f / 6.0f), del.l)};   // sin(delta)
    const float4 T = tab[idx];                            // cos + 3, its low part, sin + 3, its low part
    const float C = T.x - 3.0f, S = T.z - 3.0f;           // exact
    {
        const float s1 = fmaf(-S, sd.h, T.x), t1 = s1 - T.x, l1 = fmaf(-S, sd.h, -t1);
        const float s2 = fmaf(C, cm.h, s1), t2 = s2 - s1, l2 = fmaf(C, cm.h, -t2);
        float l = l1 + l2;
        l = fmaf(C, cm.l, l);
        l = fmaf(T.y, cm.h, l);
        l = fmaf(-S, sd.l, l);
        l = fmaf(-T.w, sd.h, l);
        cs = {s2 - 3.0f, l + T.y};
    }
    {
        const float s1 = fmaf(C, sd.h, T.z), t1 = s1 - T.z, l1 = fmaf(C, sd.h, -t1);
        const float s2 = fmaf(S, cm.h, s1), t2 = s2 - s1, l2 = fmaf(S, cm.h, -t2);
        float l = l1 + l2;
        l = fmaf(S, cm.l, l);
        l = fmaf(T.w, cm.h, l);
        l = fmaf(C, sd.l, l);
        l = fmaf(T.y, sd.h, l);
        sn = {s2 - 3.0f, l + T.w};
    }
}

// What the two directions of a pair share.
struct DflGeom {
    dd dx, dy, dz, ir2, kr, Er, Ei;
    float mr;                          // grid for n.d
};

// (W = 1: E times the weight w of the source; 2: E times w.h, a power of two)
template <int W>
__device__ __forceinline__ DflGeom dfl_geom(dd tx, dd ty, dd tz, float4 A4, float4 B4, dd w,
                                            const float4 *__restrict__ tab, const DflConst &K)
{
    DflGeom G;
    // d = x_i - x_j
    G.dx = sub(tx, {A4.x, B4.x});
    G.dy = sub(ty, {A4.y, B4.y});
    G.dz = sub(tz, {A4.z, B4.z});
    // r^2 from exact squares; the sums of the positive squares in fast_two_sum order
    const float px = G.dx.h * G.dx.h, py = G.dy.h * G.dy.h, pz = G.dz.h * G.dz.h;
    const float ex = fmaf(G.dx.h, G.dx.h, -px), ey = fmaf(G.dy.h, G.dy.h, -py), ez = fmaf(G.dz.h, G.dz.h, -pz);
    const float cr = fmaf(G.dx.h, G.dx.l, fmaf(G.dy.h, G.dy.l, G.dz.h * G.dz.l));
    const float m1 = fmaxf(px, py), l1 = fminf(px, py);
    const float s1 = m1 + l1, e1 = l1 - (s1 - m1);
    const float m2 = fmaxf(s1, pz), l2 = fminf(s1, pz);
    const float s2 = m2 + l2, e2 = l2 - (s2 - m2);
    const dd r2 = norm({s2, fmaf(2.0f, cr, (e1 + e2) + ((ex + ey) + ez))});
    // 1/r: hardware estimate y0, Halley step y0 (1 + e/2 + 3 e^2/8), e = 1 - r^2 y0^2
    const float y0 = rsqrtf(r2.h);
    const float q0 = y0 * y0, q0e = fmaf(y0, y0, -q0);
    const float u = r2.h * q0;
    const float ue = fmaf(r2.l, q0, fmaf(r2.h, q0e, fmaf(r2.h, q0, -u)));
    const float e = (1.0f - u) - ue;
    const dd ir = norm({y0, y0 * e * fmaf(e, 0.375f, 0.5f)});
    // r = rh + (r^2 - rh^2) / (2 r): rh is within an ulp of r, so the next term is below 2^-49 r
    const float rh = r2.h * ir.h;
    const float rr = fmaf(-rh, rh, r2.h) + r2.l;
    const dd r = {rh, rr * (0.5f * ir.h)};
    G.mr = dfl_magic_of(rh);
    G.ir2 = mul(ir, ir);
    G.kr = mul(K.kappa, r);
    dd cs, sn;
    dfl_cis(K.no_phase ? dd{0.f, 0.f} : r, tab, cs, sn);
    const dd iw = W == 1 ? mul(ir, w) : W == 2 ? dd{ir.h * w.h, ir.l * w.h} : ir;
    G.Er = mul(cs, iw);
    G.Ei = mul(sn, iw);
    return G;
}

// X = n.d / r^2 on the grid of r
__device__ __forceinline__ dd dfl_projection(dd nx, dd ny, dd nz, const DflGeom &G)
{
    const float s1 = fmaf(nx.h, G.dx.h, G.mr), t1 = s1 - G.mr, l1 = fmaf(nx.h, G.dx.h, -t1);
    const float s2 = fmaf(ny.h, G.dy.h, s1), t2 = s2 - s1, l2 = fmaf(ny.h, G.dy.h, -t2);
    const float s3 = fmaf(nz.h, G.dz.h, s2), t3 = s3 - s2, l3 = fmaf(nz.h, G.dz.h, -t3);
    float l = (l1 + l2) + l3;
    l = fmaf(nx.h, G.dx.l, l);
    l = fmaf(nx.l, G.dx.h, l);
    l = fmaf(ny.h, G.dy.l, l);
    l = fmaf(ny.l, G.dy.h, l);
    l = fmaf(nz.h, G.dz.l, l);
    l = fmaf(nz.l, G.dz.h, l);
    const dd nd = {s3 - G.mr, l};
    dd X = mul(nd, G.ir2);
    X.l = fmaf(nd.l, G.ir2.l, X.l);
    return X;
}

// G = E [X - i (kr X + eta')]
__device__ __forceinline__ void dfl_kernel_value(const DflGeom &G, dd X, const DflConst &K, dd &gr, dd &gi)
{
    const float s = fmaf(G.kr.h, X.h, K.eta_m), t = s - K.eta_m;
    float l = fmaf(G.kr.h, X.h, -t) + K.eta_r;
    l = fmaf(G.kr.h, X.l, l);
    l = fmaf(G.kr.l, X.h, l);
    const dd B = norm({s - K.mb, l});                      // its products with E's low part count
    gr = add(mul(G.Er, X), mul(G.Ei, B));
    gi = sub(mul(G.Ei, X), mul(G.Er, B));
}

DflConst dfl_constants(const hzb_ctx *c);
hzb_status ensure_dfl(hzb_ctx *c);
hzb_status dfl_split_reduce(hzb_ctx *c, size_t n, int nsplit, const double2 *part, double2 *y);

}  // namespace hzb
