// pfc_pair.cuh -- two voxels at a time: packed FP32 arithmetic (one
// instruction on two floats in a 64-bit register) and eq. Feps with its local
// reverse mode on a pair of voxels.
//
// The FP32 sweep is bound by instruction issue, not by the FP32 pipe: a third
// of its instructions are loads, stores, addresses and barriers.  A packed
// multiply-add occupies the pipe for as long as two scalar ones (measured: the
// same FLOP rate) but takes one issue slot, and the loads and addresses of a
// pair are shared, so the same voxels need about half the slots.
#pragma once

#include "pfc_device.cuh"
#include "pfc_log1p.h"

namespace pfc {

struct __align__(8) F2 {
    unsigned long long b;    // low word: the first voxel
};

__device__ __forceinline__ F2 pk(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.b) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ F2 dup(float x) { return pk(x, x); }
__device__ __forceinline__ float lo(F2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.b));
    return x;
}
__device__ __forceinline__ float hi(F2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.b));
    return y;
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b)
{
    F2 r;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 fma_(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r.b) : "l"(a.b), "l"(b.b), "l"(c.b));
    return r;
}

// Half the cotangents with respect to the raw stencil values (see Cot) of a
// pair of voxels (V = F2) or one FP64 voxel (V = double); the mixed ones
// without their factor 1/2 (each feeds M_cd and M_dc with the four-point
// difference's 1/4).
template <class V>
struct CotH {
    V u, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz;
};
using Cot2 = CotH<F2>;

// a number as a value of V; 1 / sqrt
template <class V> __device__ __forceinline__ V bc(double x);
template <> __device__ __forceinline__ F2 bc<F2>(double x) { return dup((float)x); }
template <> __device__ __forceinline__ double bc<double>(double x) { return x; }
__device__ __forceinline__ F2 bcv(F2, float x) { return dup(x); }
__device__ __forceinline__ double bcv(double, double x) { return x; }
__device__ __forceinline__ F2 rsq(F2 a) { return pk(rsqrtf(lo(a)), rsqrtf(hi(a))); }
__device__ __forceinline__ double rsq(double a) { return rsqrt(a); }

// Coefficients of eq. Feps and the stencil scales as pairs, for the general
// form, formed once per run (2 c2 is not: without its registers the batched
// step spills 92/144 bytes a thread, stores/loads, instead of 124/192, 24 mixed
// problems 5.8 -> 5.5 ms for 16 steps).
struct Coef2 {
    F2 c1, c2, c3, c4, c5, c6, c6x2, kd, ko, ko2, sg, nsg, ie, xi2;
    F2 c7, c7x2, th0, th1, th2;       // orientation term (ORIENT)
    float xi, xi64, inv_xi, rthr;
    int well;
};
__device__ __forceinline__ Coef2 coef2(const Coef<float>& C)
{
    Coef2 P;
    P.c1 = dup(C.c1); P.c2 = dup(C.c2); P.c3 = dup(C.c3); P.c4 = dup(C.c4); P.c5 = dup(C.c5); P.c6 = dup(C.c6);
    P.c6x2 = dup(C.c6x2);
    P.c7 = dup(C.c7); P.c7x2 = dup(2.0f * C.c7); P.th0 = dup(C.th0); P.th1 = dup(C.th1); P.th2 = dup(C.th2);
    P.kd = dup(C.kd); P.ko = dup(C.ko); P.ko2 = dup(C.ko2); P.sg = dup(C.sg); P.nsg = dup(-C.sg);
    P.ie = dup(C.inv_eps); P.xi2 = dup(C.xi2);
    P.xi = C.xi; P.xi64 = 64.0f * C.xi; P.inv_xi = C.inv_xi; P.rthr = C.rthr;
    P.well = C.well;
    return P;
}

__device__ __forceinline__ float ex2_(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

struct PairArith {   // for log1p01
    using V = F2;
    static __device__ __forceinline__ F2 c(float x) { return dup(x); }
    static __device__ __forceinline__ F2 fma(F2 a, F2 b, F2 x) { return fma_(a, b, x); }
};

// sqrt(P(D)) and d sqrt(P) / dD of both voxels (softplus_, one reciprocal
// square root for both; 0 where P underflows to 0), without branches: where
// softplus_ drops the correction (|D| > 64 xi) ex is set to 0.
__device__ __forceinline__ void root_softplus(float D0, float D1, const Coef2& C, F2& r, F2& rp)
{
    const float a0 = fabsf(D0), a1 = fabsf(D1);
    const F2 t = pk(a0, a1) * dup(-C.inv_xi) * dup(1.4426950408889634f);
    float e0 = ex2_(lo(t)), e1 = ex2_(hi(t));
    e0 = a0 > C.xi64 ? 0.0f : e0;
    e1 = a1 > C.xi64 ? 0.0f : e1;
    const F2 ex = pk(e0, e1), den = ex + dup(1.0f);
    const F2 inv = pk(__fdividef(1.0f, lo(den)), __fdividef(1.0f, hi(den)));
    const F2 exi = ex * inv;
    const F2 P = fma_(dup(C.xi), log1p01<PairArith>(ex), pk(fmaxf(D0, 0.0f), fmaxf(D1, 0.0f)));
    const F2 Pp = pk(D0 >= 0.0f ? lo(inv) : lo(exi), D1 >= 0.0f ? hi(inv) : hi(exi));
    const F2 rs = pk(rsqrtf(fmaxf(lo(P), 1e-37f)), rsqrtf(fmaxf(hi(P), 1e-37f)));
    r = P * rs;
    rp = dup(0.5f) * Pp * rs;
}

// voxel_eval's eq. Meps path on a pair: the same operations in the same order
// and rounding (D's last bits decide sqrt(D+) at the kink); ct.dx, dy, dz come
// without the stencil scale sg.
// ORIENT adds the orientation term of Sec. 5.2 (see voxel_eval).
// refine(h): D of the pair's voxel h (0 or 1) in double-float.
template <bool GRAD, bool ORIENT, class Refine>
__device__ __forceinline__ F2 pair_eval(const Coef2& C, F2 u0, F2 dx, F2 dy, F2 dz, F2 hxx, F2 hyy, F2 hzz, F2 hxy,
                                        F2 hxz, F2 hyz, Cot2& ct, const Refine& refine)
{
    const F2 one = dup(1.0f), two = dup(2.0f), mone = dup(-1.0f), mtwo = dup(-2.0f);
    const F2 Gx = dx * C.sg, Gy = dy * C.sg, Gz = dz * C.sg;
    const F2 g2 = fma_(Gx, Gx, fma_(Gy, Gy, Gz * Gz));
    const F2 rho = g2 + C.xi2;
    const F2 iq = pk(rsqrtf(lo(rho)), rsqrtf(hi(rho)));
    const F2 q = rho * iq;
    const F2 irho = iq * iq;
    F2 wp, wpp;              // W'(u), W''(u)
    if (C.well == 0) {
        const F2 t = fma_(u0 * mone, u0, u0);                 // u (1 - u)
        wp = (t * two) * fma_(u0, mtwo, one);
        wpp = fma_(t, dup(-12.0f), two);                      // 2 (1 - 6u + 6u^2)
    } else {
        const F2 uu = u0 * u0;
        wp = fma_(uu, u0, u0 * mone);
        wpp = fma_(dup(3.0f) * u0, u0, mone);
    }
    const F2 wr = wp * C.ie * irho;                           // (W'/eps) / rho
    const F2 wx = wr * Gx, wy = wr * Gy, wz = wr * Gz;
    const F2 Mxx = fma_(C.kd, hxx, wx * Gx), Myy = fma_(C.kd, hyy, wy * Gy), Mzz = fma_(C.kd, hzz, wz * Gz);
    const F2 Mxy = fma_(C.ko, hxy, wx * Gy), Mxz = fma_(C.ko, hxz, wx * Gz), Myz = fma_(C.ko, hyz, wy * Gz);
    const F2 Tr = Mxx + Myy + Mzz;
    const F2 off = fma_(Mxy, Mxy, fma_(Mxz, Mxz, Myz * Myz));
    const F2 S = fma_(Mxx, Mxx, fma_(Myy, Myy, fma_(Mzz, Mzz, off + off)));
    const F2 t2 = Tr * Tr;
    const F2 c4q = C.c4 * q;
    const F2 a3 = fma_(C.c3, Tr, C.c5 * q);
    const F2 nt2 = t2 * mone;
    const F2 t2e = fma_(Tr, Tr, nt2);                         // the rounding error of T^2, put back
    const F2 D = fma_(two, S, nt2) - t2e;
    const F2 scale = fma_(two, S, t2);
    float D0 = lo(D), D1 = hi(D);
    const bool n0 = lo(a3) != 0.0f && lo(scale) > C.rthr * fmax_nan_(fabsf(D0), C.xi);
    const bool n1 = hi(a3) != 0.0f && hi(scale) > C.rthr * fmax_nan_(fabsf(D1), C.xi);
    if (n0 || n1) {
        if (n0) D0 = refine(0);
        if (n1) D1 = refine(1);
    }
    F2 r, rp;
    root_softplus(D0, D1, C, r, rp);
    F2 e = fma_(C.c1, S, fma_(C.c2, t2, fma_(a3, r, fma_(c4q, Tr, C.c6 * g2))));
    F2 tg;
    if constexpr (ORIENT) {
        tg = fma_(C.th0, Gx, fma_(C.th1, Gy, C.th2 * Gz));
        e = fma_(C.c7 * tg, tg, e);
    }
    if constexpr (!GRAD) return e;
    const F2 k = a3 * rp;                                     // de/dD
    const F2 dT = fma_(C.c2, Tr + Tr, fma_(C.c3, r, fma_(C.c4, q, (Tr * mtwo) * k)));
    const F2 dq = fma_(C.c4, Tr, C.c5 * r);
    const F2 s2 = two * fma_(two, k, C.c1);
    // Lambda = de/dM = 2 dS M + dT I
    const F2 Lxx = fma_(s2, Mxx, dT), Lyy = fma_(s2, Myy, dT), Lzz = fma_(s2, Mzz, dT);
    const F2 Lxy = s2 * Mxy, Lxz = s2 * Mxz, Lyz = s2 * Myz;
    const F2 LGx = fma_(Lxx, Gx, fma_(Lxy, Gy, Lxz * Gz));
    const F2 LGy = fma_(Lxy, Gx, fma_(Lyy, Gy, Lyz * Gz));
    const F2 LGz = fma_(Lxz, Gx, fma_(Lyz, Gy, Lzz * Gz));
    const F2 GLG = fma_(Gx, LGx, fma_(Gy, LGy, Gz * LGz));
    ct.u = wpp * C.ie * GLG * irho;
    const F2 al = wr * two;
    const F2 be = fma_((wr * mtwo) * GLG, irho, fma_(dq, iq, C.c6x2));
    ct.dx = fma_(al, LGx, be * Gx);
    ct.dy = fma_(al, LGy, be * Gy);
    ct.dz = fma_(al, LGz, be * Gz);
    if constexpr (ORIENT) {
        const F2 ot = C.c7x2 * tg;
        ct.dx = fma_(ot, C.th0, ct.dx);
        ct.dy = fma_(ot, C.th1, ct.dy);
        ct.dz = fma_(ot, C.th2, ct.dz);
    }
    ct.hxx = C.kd * Lxx; ct.hyy = C.kd * Lyy; ct.hzz = C.kd * Lzz;
    ct.hxy = C.ko2 * Lxy; ct.hxz = C.ko2 * Lxz; ct.hyz = C.ko2 * Lyz;   // Hess_cd feeds M_cd and M_dc
    return e;
}

// The density and half its cotangents (Cot2) for c3 = c5 = 0, on the raw differences d = grad u / sg: with
// M = kd N and G = sg d, N_cc = h_cc + w d_c d_c and N_cd = h_cd / 4 + w d_c
// d_d, w = W' / (eps kd) / (|d|^2 + xi^2 / sg^2); e = n1 ||N||^2 + n2 T^2 +
// 2 n4 q T + n6 |d|^2 with q = sqrt(|d|^2 + xi^2 / sg^2).  No stencil scale is
// applied and no second difference multiplied: 14 products fewer.
template <bool GRAD, class V, class T>
__device__ __forceinline__ V eval_sym(const Coef<T>& C, V u0, V dx, V dy, V dz, V hxx, V hyy, V hzz, V hxy, V hxz,
                                      V hyz, CotH<V>& ct)
{
    auto k = [&](T x) { return bcv(u0, x); };
    const V one = bc<V>(1.0), quarter = bc<V>(0.25), n1 = k(C.n1);
    const V g2 = fma_(dx, dx, fma_(dy, dy, dz * dz));
    const V rho = g2 + k(C.nx2);
    const V iq = rsq(rho);
    const V q = rho * iq;
    const V irho = iq * iq;
    V wp, wpk;              // W'(u) / wB K, W''(u) K
    if (C.well == 0) {
        const V v = one - u0;
        const V t = u0 * v;                                  // W' = 2 t (1 - 2u), W'' = 2 - 12 t
        wp = t * (v - u0);
        wpk = fma_(t, k(C.wA), k(C.wB));
    } else {
        const V uu = u0 * u0;                                // W' = -u (1 - u^2), W'' = 3 u^2 - 1
        wp = u0 * (one - uu);
        wpk = fma_(uu, k(C.wA), k(C.wB));
    }
    const V w = wp * k(C.wB) * irho;
    const V wx = w * dx, wy = w * dy, wz = w * dz;
    const V Nxx = fma_(wx, dx, hxx), Nyy = fma_(wy, dy, hyy), Nzz = fma_(wz, dz, hzz);
    const V Nxy = fma_(quarter, hxy, wx * dy), Nxz = fma_(quarter, hxz, wx * dz), Nyz = fma_(quarter, hyz, wy * dz);
    const V Tr = Nxx + Nyy + Nzz;
    const V off = fma_(Nxy, Nxy, fma_(Nxz, Nxz, Nyz * Nyz));
    const V S = fma_(Nxx, Nxx, fma_(Nyy, Nyy, fma_(Nzz, Nzz, off + off)));
    const V q4 = k(C.n4) * q;
    const V dT = fma_(k(C.n2), Tr, q4);                    // half of de/dT
    const V e = fma_(n1, S, fma_(Tr, dT + q4, k(C.n6) * g2));
    if constexpr (!GRAD) return e;
    const V Lxx = fma_(n1, Nxx, dT), Lyy = fma_(n1, Nyy, dT), Lzz = fma_(n1, Nzz, dT);
    const V Lxy = n1 * Nxy, Lxz = n1 * Nxz, Lyz = n1 * Nyz;
    const V LGx = fma_(Lxx, dx, fma_(Lxy, dy, Lxz * dz));
    const V LGy = fma_(Lxy, dx, fma_(Lyy, dy, Lyz * dz));
    const V LGz = fma_(Lxz, dx, fma_(Lyz, dy, Lzz * dz));
    const V GLG = fma_(dx, LGx, fma_(dy, LGy, dz * LGz));
    ct.u = wpk * GLG * irho;
    const V al = w + w;
    const V be = fma_(k(C.n4) * Tr, iq, k(C.n6)) - al * GLG * irho;
    ct.dx = fma_(al, LGx, be * dx);
    ct.dy = fma_(al, LGy, be * dy);
    ct.dz = fma_(al, LGz, be * dz);
    ct.hxx = Lxx; ct.hyy = Lyy; ct.hzz = Lzz;
    ct.hxy = Lxy; ct.hxz = Lxz; ct.hyz = Lyz;
    return e;
}

}  // namespace pfc
