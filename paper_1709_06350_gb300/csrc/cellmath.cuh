// cellmath.cuh -- per-cell arithmetic of the reconstruction equation, for
// T = double or float.  Every kernel that touches the discrete operator goes
// through these functions.
//
//   Hessian stencils          Sec. II.A.1, eq. discrete_examples
//   cubic s^3 + p s + q = 0   Sec. II, eqs. final_PDE / final_PDE2, with the
//                             traceless part Hbar of eq. transformation_derivatives
//   physical root             eq. root, read as the LARGEST real root
//   point update              eq. update, dL/dtheta_c = -6/h^2
#pragma once

#include "common.cuh"

namespace recon {

__device__ __forceinline__ double m_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float m_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double m_cbrt(double x) { return cbrt(x); }
__device__ __forceinline__ float m_cbrt(float x) { return cbrtf(x); }
__device__ __forceinline__ double m_acos(double x) { return acos(x); }
__device__ __forceinline__ float m_acos(float x) { return acosf(x); }
__device__ __forceinline__ double m_cos(double x) { return cos(x); }
__device__ __forceinline__ float m_cos(float x) { return cosf(x); }
__device__ __forceinline__ double m_abs(double x) { return fabs(x); }
__device__ __forceinline__ float m_abs(float x) { return fabsf(x); }

// The 19-point neighbourhood of a cell: centre, 6 faces, 12 edges (no corners).
template <typename T>
struct Nb19 {
    T c;
    T xp, xm, yp, ym, zp, zm;
    T xpyp, xmym, xmyp, xpym;  // (i+-1, j+-1, k)
    T ypzp, ymzm, ymzp, ypzm;  // (i, j+-1, k+-1)
    T xpzp, xmzm, xmzp, xpzm;  // (i+-1, j, k+-1)
};

// 32-bit offsets: grids are limited to N <= 1024 (N^3 < 2^32).
template <typename T, typename P>
__device__ __forceinline__ Nb19<T> load19(P a, int N, int i, int j, int k)
{
    const unsigned n = (unsigned)N, nn = n * n;
    const unsigned ri = (unsigned)i * nn, rip = (unsigned)wp(i, N) * nn, rim = (unsigned)wm(i, N) * nn;
    const unsigned cj = (unsigned)j * n, cjp = (unsigned)wp(j, N) * n, cjm = (unsigned)wm(j, N) * n;
    const unsigned kk = (unsigned)k, kp = (unsigned)wp(k, N), km = (unsigned)wm(k, N);
    Nb19<T> v;
    v.c = a[ri + cj + kk];
    v.xp = a[rip + cj + kk];
    v.xm = a[rim + cj + kk];
    v.yp = a[ri + cjp + kk];
    v.ym = a[ri + cjm + kk];
    v.zp = a[ri + cj + kp];
    v.zm = a[ri + cj + km];
    v.xpyp = a[rip + cjp + kk];
    v.xmym = a[rim + cjm + kk];
    v.xmyp = a[rim + cjp + kk];
    v.xpym = a[rip + cjm + kk];
    v.ypzp = a[ri + cjp + kp];
    v.ymzm = a[ri + cjm + km];
    v.ymzp = a[ri + cjm + kp];
    v.ypzm = a[ri + cjp + km];
    v.xpzp = a[rip + cj + kp];
    v.xmzm = a[rim + cj + km];
    v.xmzp = a[rim + cj + kp];
    v.xpzm = a[rip + cj + km];
    return v;
}

// Off-diagonal Hessian entries (4-point edge stencils / (4 h^2)).
template <typename T>
__device__ __forceinline__ void mixed(const Nb19<T> &n, T q4, T &hxy, T &hyz, T &hxz)
{
    hxy = ((n.xpyp + n.xmym) - (n.xmyp + n.xpym)) * q4;
    hyz = ((n.ypzp + n.ymzm) - (n.ymzp + n.ypzm)) * q4;
    hxz = ((n.xpzp + n.xmzm) - (n.xmzp + n.xpzm)) * q4;
}

// Coefficients of the cell cubic s^3 + p s + q = 0 with s = 3 + lap theta:
//   Hbar_aa = (2 S_a - S_b - S_c) / (3 h^2)  (S_a = sum of the two face
//   neighbours along a; the centre cancels, as the paper notes),
//   p = -(9/2) tr(Hbar^2),  q = 27 det(Hbar) - 27 rhs.
template <typename T>
__device__ __forceinline__ void cubic_coeffs(const Nb19<T> &n, T ih2, T rhs, T &s, T &p, T &q)
{
    const T X = n.xp + n.xm, Y = n.yp + n.ym, Z = n.zp + n.zm;
    const T third = ih2 * T(1.0 / 3.0);
    const T bxx = (T(2) * X - Y - Z) * third;
    const T byy = (T(2) * Y - Z - X) * third;
    const T bzz = (T(2) * Z - X - Y) * third;
    T hxy, hyz, hxz;
    mixed(n, ih2 * T(0.25), hxy, hyz, hxz);
    s = T(3) + ((X + Y + Z) - T(6) * n.c) * ih2;
    const T tr2 = bxx * bxx + byy * byy + bzz * bzz + T(2) * (hxy * hxy + hyz * hyz + hxz * hxz);
    const T detb = bxx * (byy * bzz - hyz * hyz) - hxy * (hxy * bzz - hyz * hxz)
                 + hxz * (hxy * hyz - byy * hxz);
    p = T(-4.5) * tr2;
    q = T(27) * detb - T(27) * rhs;
}

// det(I + H) at the cell (first-row expansion).
template <typename T>
__device__ __forceinline__ T det_IH(const Nb19<T> &n, T ih2)
{
    const T axx = T(1) + ((n.xp + n.xm) - T(2) * n.c) * ih2;
    const T ayy = T(1) + ((n.yp + n.ym) - T(2) * n.c) * ih2;
    const T azz = T(1) + ((n.zp + n.zm) - T(2) * n.c) * ih2;
    T hxy, hyz, hxz;
    mixed(n, ih2 * T(0.25), hxy, hyz, hxz);
    return axx * (ayy * azz - hyz * hyz) - hxy * (hxy * azz - hyz * hxz)
         + hxz * (hxy * hyz - ayy * hxz);
}

// adj(I + H): (xx, yy, zz, xy, yz, xz); J v = sum adj_ab D_ab v.
template <typename T>
struct Cof {
    T xx, yy, zz, xy, yz, xz;
};
template <typename T>
__device__ __forceinline__ Cof<T> cofactors(const Nb19<T> &n, T ih2)
{
    const T axx = T(1) + ((n.xp + n.xm) - T(2) * n.c) * ih2;
    const T ayy = T(1) + ((n.yp + n.ym) - T(2) * n.c) * ih2;
    const T azz = T(1) + ((n.zp + n.zm) - T(2) * n.c) * ih2;
    T hxy, hyz, hxz;
    mixed(n, ih2 * T(0.25), hxy, hyz, hxz);
    Cof<T> a;
    a.xx = ayy * azz - hyz * hyz;
    a.yy = axx * azz - hxz * hxz;
    a.zz = axx * ayy - hxy * hxy;
    a.xy = hxz * hyz - hxy * azz;
    a.yz = hxy * hxz - axx * hyz;
    a.xz = hxy * hyz - hxz * ayy;
    return a;
}

// sum_ab adj_ab D_ab v at a cell, from v's 19-point neighbourhood.
template <typename T>
__device__ __forceinline__ T jac_apply(const Cof<T> &a, const Nb19<T> &v, T ih2)
{
    const T dxx = ((v.xp + v.xm) - T(2) * v.c) * ih2;
    const T dyy = ((v.yp + v.ym) - T(2) * v.c) * ih2;
    const T dzz = ((v.zp + v.zm) - T(2) * v.c) * ih2;
    T dxy, dyz, dxz;
    mixed(v, ih2 * T(0.25), dxy, dyz, dxz);
    return a.xx * dxx + a.yy * dyy + a.zz * dzz + T(2) * (a.xy * dxy + a.yz * dyz + a.xz * dxz);
}

// Largest real root of s^3 + p s + q (p <= 0 for a symmetric Hbar).
//   Delta >= 0: u = cbrt(-q/2 + sgn(-q/2) sqrt(Delta)), s = u - p/(3u)
//   Delta <  0: s = 2 sqrt(-p/3) cos(sigma/3), cos sigma = (3q/2p) sqrt(-3/p)
template <typename T>
__device__ __forceinline__ T largest_root(T p, T q)
{
    const T D = q * q * T(0.25) + p * p * p * T(1.0 / 27.0);
    if (D >= T(0)) {
        const T a = -q * T(0.5);
        const T u = m_cbrt(a + (a >= T(0) ? m_sqrt(D) : -m_sqrt(D)));
        return u == T(0) ? T(0) : u - p / (T(3) * u);
    }
    T arg = (T(3) * q / (T(2) * p)) * m_sqrt(T(-3) / p);
    arg = arg > T(1) ? T(1) : (arg < T(-1) ? T(-1) : arg);
    return T(2) * m_sqrt(-p * T(1.0 / 3.0)) * m_cos(m_acos(arg) * T(1.0 / 3.0));
}

template <typename T>
__device__ __forceinline__ T root_polished(T p, T q)
{
    T sn = largest_root(p, q);
    const T fp = T(3) * sn * sn + p;
    if (fp > T(0)) sn = sn - (sn * sn * sn + p * sn + q) / fp;
    return sn;
}

// Eq. update: theta_c - (h^2/6)(s_new - s).
//   rule 1: s_new = largest root (the paper's update), Newton-polished;
//   rule 0: one Newton step on the cubic from s, taken only right of the
//           local minimum of f (s > sqrt(-p/3)) and kept only if |f| does not
//           grow; else rule 1.
// |f| after the step is taken in the cancellation-free form
// f(s + d) = d^2 (3 s + d) for the Newton step d = -f / f', so the test is
// |d| |3 s + d| <= f'; recomputing f(s + d) near convergence gives rounding
// noise, which rejects good steps at random (and sent whole warps through the
// root of the cubic: an FP64 sweep of 128^3 took 461 us, 209 us in this form;
// at one FP64 operation per 64 FP32 ones its ~50 operations are ~197 us).

// FP32, on the cubic s^3 + p s + q; the quotient is the fast reciprocal form
// (2 ulp), whose result the defect correction refines
__device__ __forceinline__ float cell_update(const Nb19<float> &n, float rhs, float ih2, float h2_6, int rule)
{
    float s, p, q, sn;
    cubic_coeffs(n, ih2, rhs, s, p, q);
    bool done = false;
    if (rule == 0 && s > 0.0f && 3.0f * s * s > -p) {
        const float f = s * s * s + p * s + q;
        const float fp = 3.0f * s * s + p;
        const float quot = __fdividef(f, fp);
        sn = s - quot;
        done = fabsf(quot * (3.0f * s - quot)) <= fp;
    }
    if (!done) sn = root_polished(p, q);
    return n.c - h2_6 * (sn - s);
}

// a / b within 1 ulp, where b is positive and b, 1 / b and the quotient are
// normal numbers (b from 2^-1022 to 2^1022; beyond, the reciprocal is flushed
// to zero or infinity).  Newton's iteration for 1 / b, with Markstein's
// remainder step for the quotient: the hardware's reciprocal approximation, one
// Newton step on 1 / b (to ~40 bits) and one on the quotient, whose remainder
// is exact in one fma.  Four FP64 operations and no branch; FP64 operations are
// what the FP64 smoother waits for.
__device__ __forceinline__ double div_pos(double a, double b)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    r = fma(r, fma(-b, r, 1.0), r);
    const double q = a * r;
    return fma(fma(-b, q, a), r, q);
}

// Rule 1 from A = I + H theta: the cubic of the traceless part, its largest
// root; returns theta_c - (h^2/6)(root - tr A).  Out of line: rare under rule 0.
static __device__ __noinline__ double root_update(double theta_c, double axx, double ayy, double azz, double hxy,
                                                  double hyz, double hxz, double rhs, double h2_6)
{
    const double s = axx + ayy + azz, third = s * (1.0 / 3.0);
    const double bxx = axx - third, byy = ayy - third, bzz = azz - third;
    const double tr2 = bxx * bxx + byy * byy + bzz * bzz + 2.0 * (hxy * hxy + hyz * hyz + hxz * hxz);
    const double detb = bxx * (byy * bzz - hyz * hyz) - hxy * (hxy * bzz - hyz * hxz)
                      + hxz * (hxy * hyz - byy * hxz);
    return theta_c - h2_6 * (root_polished(-4.5 * tr2, 27.0 * detb - 27.0 * rhs) - s);
}

// FP64, on A = I + H theta directly: with s = tr A and S = tr adj A the cubic
// is f = 27 (det A - rhs) with f' = 9 S, so Newton's step is
// tau = (det A - rhs) / S, theta_c += (h^2/2) tau (every diagonal entry of A
// moves by -tau), kept when s > 0, S > 0 and |tau| |s - tau| <= S.  ~50 FP64
// operations per cell; the tests run on the integer pipes (signs, and the
// order of the bit patterns of two non-negative numbers).  resid (nullable):
// rhs - det A.
__device__ __forceinline__ double cell_update(const Nb19<double> &n, double rhs, double ih2, double h2_6, int rule,
                                              double *resid = nullptr)
{
    const double axx = fma(fma(-2.0, n.c, n.xp + n.xm), ih2, 1.0);
    const double ayy = fma(fma(-2.0, n.c, n.yp + n.ym), ih2, 1.0);
    const double azz = fma(fma(-2.0, n.c, n.zp + n.zm), ih2, 1.0);
    double hxy, hyz, hxz;
    mixed(n, ih2 * 0.25, hxy, hyz, hxz);
    const double cxx = fma(-hyz, hyz, ayy * azz);
    const double cyy = fma(-hxz, hxz, axx * azz);
    const double czz = fma(-hxy, hxy, axx * ayy);
    const double cxy = fma(hxz, hyz, -(hxy * azz));
    const double cxz = fma(hxy, hyz, -(hxz * ayy));
    const double F = fma(axx, cxx, fma(hxy, cxy, fma(hxz, cxz, -rhs)));
    if (resid) *resid = -F;
    const double S = cxx + cyy + czz, s = axx + ayy + azz;
    const double tau = div_pos(F, S), u = tau * (s - tau);
    const long long ub = __double_as_longlong(u) & 0x7fffffffffffffffll;
    if (rule == 0 && __double_as_longlong(s) > 0 && ub <= __double_as_longlong(S))   // (u a NaN: false)
        return fma(tau, 3.0 * h2_6, n.c);
    return root_update(n.c, axx, ayy, azz, hxy, hyz, hxz, rhs, h2_6);
}

}  // namespace recon
