// One multipole interaction in the wide element types (double, double-float).
//
// Both types are bound by their arithmetic pipe (GB300 issues one FP64
// operation for 64 FP32 ones; a double-float operation is 7 to 12 FP32
// operations), so the contraction is written for the fewest operations:
//   - the packed moments are the traceless parts of M2 and M3 themselves,
//     t2 = (3/2) T2 / h^2 and t3 = (5/2) T3 / h^3 (fmm_m2l.cu packs them).
//     Against a traceless tensor every delta term of D2, D3 and D4 vanishes,
//     so no derivative tensor of order >= 2 is formed for the source's
//     moments: with q = t2 R, s2 = R.t2.R, b = t3:RR, s3 = t3:RRR and
//     e_k = 1/r^k,
//       L0  -= m e1 + e5 s2 + e7 s3,
//       L1  += R (m e3 + 5 e7 s2) - 2 e5 q,
//       dL1 += 7 e9 s3 R - 3 e7 b                       (the source's share);
//   - what depends on the source's mass alone (orders 2 and 3 of the Taylor
//     coefficients, and the target's share of the correction,
//     -sum m D4 : M3_A / (6 M0_A)) is summed as moments m e_k R R.. of the
//     separations: those of L2 and L3 made traceless term by term, the others
//     plain, since the delta terms of D4 and the contraction with the target's
//     own third moment are linear in the sums and so are formed once per target
//     cell (finish()) instead of once per source.
// 72 operations for a leaf source and 127 for a refined one (fused
// multiply-add = 1), where evaluating the derivative tensors and contracting
// them takes about 145 and 173 (with the divide and square root of
// 1 / sqrt).  A level-6 binary (5225 sub-grids, theta 0.5), whole step: FP64
// 31.4 -> 24.4 ms (multipole kernel 26.1 -> 19.1, its FP64 pipe 91 % busy
// before and after), double-float 6.65 -> 5.48 ms; a 9-sub-grid FP64 step 968
// -> 318 us (the root over 128 CTAs).  Errors against 64 bits, level-5 binary,
// tensors / this: double-float g 1.2e-14 / 9e-15, phi 8.0e-15 / 4.4e-15, L2
// 2.0e-14 / 9e-15, L3 3.1e-14 / 1.3e-14; FP64 g 4.6e-16 / 4.6e-16, L3 1.1e-15 /
// 1.0e-15.  (L2 and L3 as plain moments, whose traces do not cancel, and sums
// normalised every 16 entries only: 3 % faster in double-float, 1.5 % in FP64,
// with L3 at 4.7e-14 and 1.2e-15.)
#pragma once

#include "fmm_convert.cuh"
#include "fmm_dfloat.cuh"
#include "fmm_tensor.cuh"

namespace fmm {

// products that the compiler may not fuse into a following sum, so that every
// kernel an interaction is compiled into rounds it alike; a small constant
// times a value; twice a value (exact)
__device__ __forceinline__ double product(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ dfloat product(dfloat a, dfloat b) { return mul_u(a, b); }
// (mul_u, fmm_dfloat.cuh: products that only enter further products)
__device__ __forceinline__ double mul_u(double a, double b) { return a * b; }
__device__ __forceinline__ double scaled(float c, double v) { return __dmul_rn(double(c), v); }
__device__ __forceinline__ dfloat scaled(float c, dfloat v) { return c * v; }
__device__ __forceinline__ double twice(double v) { return v + v; }
__device__ __forceinline__ dfloat twice(dfloat v) { return dfloat(v.hi + v.hi, v.lo + v.lo); }
// n a + b, n a small whole number
__device__ __forceinline__ double multiple(float n, double a, double b) { return fma(double(n), a, b); }
__device__ __forceinline__ dfloat multiple(float n, dfloat a, dfloat b)
{
    const float p = n * a.hi, e = fmaf(n, a.lo, fmaf(n, a.hi, -p));
    return renorm(add_u(dfloat(p, e), b));
}

// 1/sqrt(v): the hardware's float estimate y0 of a float of v, refined by the
// binomial series of (1 - e)^(-1/2), e = 1 - v y0^2 (|e| < 2^-21): with the
// terms 1 + e/2 + 3 e^2/8 the relative truncation is below 5/16 e^3 < 2^-64.
// y0^2 is exact in double (24-bit y0).  Five FP64 operations, the
// conversions on the integer pipe.  v is a squared distance in cell widths:
// inside float's normal range.
__device__ __forceinline__ double rsqrt_wide(double v)
{
    const double y = f2d_bits(rsqrt_ftz(d2f_trunc(v)));
    const double e = fma(-v, y * y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ dfloat rsqrt_wide(dfloat v) { return df_rsqrt(v); }

// x^2 + y^2 + z^2 given the three squares
__device__ __forceinline__ double wide_r2(double x, double y, double, double, double zz)
{
    return fma(x, x, fma(y, y, zz));
}
__device__ __forceinline__ dfloat wide_r2(dfloat, dfloat, dfloat xx, dfloat yy, dfloat zz)
{
    return renorm(add_u(add_u(xx, yy), zz));
}

// separation component (a - d) - e, e a whole number
__device__ __forceinline__ double wide_sep(double a, double d, float e) { return (a - d) - f2d_bits(e); }
__device__ __forceinline__ dfloat wide_sep(dfloat a, dfloat d, float e)
{
    return renorm(add_u(add_u(a, -d), dfloat(-e)));
}

// packed data of one refined source cell
template <typename T>
struct WideSrc {
    T d[3], m0;              // centre-of-mass offset / h, mass
    T t2[5];                 // xx yy xy xz yz
    T t3[7];                 // xxx xxy xxz xyy xyz yyy yyz
};

// separation R and what both halves of an interaction use of it
template <typename T>
struct WideGeo {
    T R[3], e1, e3, e5, e7, e9;
    T xx, yy, xy2, xz2, yz2;         // the mixed products doubled
    T r2, u, v;                      // xx - zz, yy - zz
    template <int ORDER>
    __device__ __forceinline__ void eval(T x, T y, T z)
    {
        R[0] = x; R[1] = y; R[2] = z;
        xx = renorm(product(x, x)); yy = renorm(product(y, y));
        const T zz = renorm(product(z, z));
        r2 = wide_r2(x, y, xx, yy, zz);
        u = xx - zz;
        v = yy - zz;
        e1 = rsqrt_wide(r2);
        const T i2 = e1 * e1;
        e3 = e1 * i2;
        e5 = e3 * i2;
        e7 = e5 * i2;
        if (ORDER == 3) e9 = e7 * i2;
        const T x2 = twice(x), y2 = twice(y);
        xy2 = mul_u(x2, y); xz2 = mul_u(x2, z); yz2 = mul_u(y2, z);
    }
};

// q = t2 R for the traceless t2
template <typename T>
__device__ __forceinline__ void wide_t2R(const T t2[5], const T R[3], T q[3])
{
    q[0] = renorm(fmadd_u(t2[3], R[2], fmadd_u(t2[2], R[1], mul_u(t2[0], R[0]))));
    q[1] = renorm(fmadd_u(t2[4], R[2], fmadd_u(t2[2], R[0], mul_u(t2[1], R[1]))));
    q[2] = renorm(fmadd_u(-(t2[0] + t2[1]), R[2], fmadd_u(t2[4], R[1], mul_u(t2[3], R[0]))));
}

// b = t3 : R R for the traceless t3 (zz eliminated)
template <typename T>
__device__ __forceinline__ void wide_t3RR(const T t3[7], const WideGeo<T> &g, T b[3])
{
    const T u = g.u, v = g.v;
    const T nxzz = t3[0] + t3[3], nyzz = t3[1] + t3[5];       // -xzz, -yzz
    b[0] = renorm(fmadd_u(t3[4], g.yz2, fmadd_u(t3[2], g.xz2, fmadd_u(t3[1], g.xy2, fmadd_u(t3[3], v, mul_u(t3[0], u))))));
    b[1] = renorm(fmadd_u(t3[6], g.yz2, fmadd_u(t3[4], g.xz2, fmadd_u(t3[3], g.xy2, fmadd_u(t3[5], v, mul_u(t3[1], u))))));
    b[2] = renorm(fmadd_u(-nyzz, g.yz2, fmadd_u(-nxzz, g.xz2, fmadd_u(t3[4], g.xy2, fmadd_u(t3[6], v, mul_u(t3[2], u))))));
}

template <typename T>
__device__ __forceinline__ T wide_dot(const T a[3], const T b[3])
{
    return renorm(fmadd_u(a[2], b[2], fmadd_u(a[1], b[1], mul_u(a[0], b[0]))));
}

// Sums of a leaf target (orders 0-1 and the correction; refined sources only)
// and, as the first part of WideAcc, of a refined one.
template <typename T, int ORDER>
struct WideLow {
    T a0, a1[3], s[3];       // -L0, L1, the source's share of the correction
                             // (over 3 at order 3)
    __device__ __forceinline__ void zero()
    {
        a0 = T(0);
#pragma unroll
        for (int i = 0; i < 3; ++i) a1[i] = s[i] = T(0);
    }
    __device__ __forceinline__ void flush()
    {
        a0 = renorm(a0);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            a1[i] = renorm(a1[i]);
            s[i] = renorm(s[i]);
        }
    }
    // a source of mass m; with MP also its moments (src.m0 is not used: a
    // warp that mixes leaf and refined sources passes m and zero moments)
    __device__ __forceinline__ void add(const WideGeo<T> &g, T me3, T m, const WideSrc<T> &src, bool mp)
    {
        // a source's terms of L0 and L1 are summed first, so that it costs one
        // rounding at the sums' magnitude
        T t0 = product(m, g.e1), f = me3, t1[3] = {T(0), T(0), T(0)};
        if (mp) {
            T q[3];
            wide_t2R(src.t2, g.R, q);
            const T s2 = wide_dot(q, g.R);
            t0 = fmadd_u(g.e5, s2, t0);
            const T k = mul_u(g.e7, s2);
            const T n2e5 = -twice(g.e5);
            if constexpr (ORDER == 3) {
                T b[3];
                wide_t3RR(src.t3, g, b);
                const T s3 = wide_dot(b, g.R);
                t0 = fmadd_u(g.e7, s3, t0);
                f = renorm(fmadd_u(T(5), k, f));
                const T c = mul_u(mul_u(g.e9, s3), T(7.0 / 3.0));
                const T ne7 = -g.e7;
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    t1[i] = mul_u(n2e5, q[i]);
                    s[i] = fmadd_u(ne7, b[i], fmadd_u(c, g.R[i], s[i]));
                }
            } else {
                const T c = scaled(5.f, k);
#pragma unroll
                for (int i = 0; i < 3; ++i) s[i] = fmadd_u(n2e5, q[i], fmadd_u(c, g.R[i], s[i]));
            }
            t0 = renorm(t0);
        }
        a0 = renorm(add_u(a0, t0));
        if (ORDER == 3 && mp) {
#pragma unroll
            for (int i = 0; i < 3; ++i) a1[i] = renorm(add_u(a1[i], renorm(fmadd_u(f, g.R[i], t1[i]))));
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) a1[i] = renorm(fmadd_u(f, g.R[i], a1[i]));
        }
    }
    __device__ __forceinline__ void correction(T S[3]) const
    {
#pragma unroll
        for (int i = 0; i < 3; ++i) S[i] = ORDER == 3 ? scaled(3.f, s[i]) : s[i];
    }
};

// Sums of a refined target: WideLow's and the mass-weighted moments of the
// separations (products of two different axes doubled, as in WideGeo).  The
// terms of L2 and L3 are made traceless one by one: as plain moments, their
// traces (sums of one sign) carried more rounding than the results have.
template <typename T, int ORDER>
struct WideAcc {
    WideLow<T, ORDER> low;
    T c2[5];                 // sum m e5 (2 xx - yy - zz, 2 yy - xx - zz, xy xz yz)
    T c3[7];                 // order 3: m e7 (x (5 xx - 3 r2), y (5 xx - r2), z (5 xx - r2),
                             // x (5 yy - r2), xyz, y (5 yy - 3 r2), z (5 yy - r2));
                             // order 2: m e7 (xxx xxy xxz xyy xyz yyy yyz)
    T more[ORDER == 3 ? 15 : 3];
    // order 3: sum m e5;  m e7 (xx yy xy xz yz);  m e9 (xxxx xxxy xxxz xxyy xxyz
    // xyyy xyyz yyyy yyyz);  order 2: m e5 (x y z)
    static constexpr int kE5 = 0, kC7 = 1, kC4 = 6, kV = 0;
    __device__ __forceinline__ void zero()
    {
        low.zero();
#pragma unroll
        for (int k = 0; k < 5; ++k) c2[k] = T(0);
#pragma unroll
        for (int k = 0; k < 7; ++k) c3[k] = T(0);
#pragma unroll
        for (int k = 0; k < (ORDER == 3 ? 15 : 3); ++k) more[k] = T(0);
    }
    // double-float: restore the canonical form (the sums take unnormalised
    // terms); called every 16 stencil entries
    __device__ __forceinline__ void flush()
    {
        low.flush();
#pragma unroll
        for (int k = 0; k < 5; ++k) c2[k] = renorm(c2[k]);
#pragma unroll
        for (int k = 0; k < 7; ++k) c3[k] = renorm(c3[k]);
#pragma unroll
        for (int k = 0; k < (ORDER == 3 ? 15 : 3); ++k) more[k] = renorm(more[k]);
    }
    __device__ __forceinline__ void add(T x, T y, T z, T m, const WideSrc<T> &src, bool mp)
    {
        WideGeo<T> g;
        g.template eval<ORDER>(x, y, z);
        const T me3 = product(m, g.e3), me5 = product(m, g.e5), me7 = mul_u(m, g.e7);
        const T two[5] = {multiple(2.f, g.u, -g.v), multiple(2.f, g.v, -g.u), g.xy2, g.xz2, g.yz2};
#pragma unroll
        for (int k = 0; k < 5; ++k) c2[k] = renorm(fmadd_u(me5, two[k], c2[k]));
        const T gx = mul_u(me7, x), gy = mul_u(me7, y);
        if constexpr (ORDER == 3) {
            const T gz = mul_u(me7, z);
            const T a = multiple(5.f, g.xx, -g.r2), b = multiple(5.f, g.yy, -g.r2);
            const T t[7] = {multiple(-2.f, g.r2, a), a, a, b, g.yz2, multiple(-2.f, g.r2, b), b};
            const T f[7] = {gx, gy, gz, gx, gx, gy, gz};
#pragma unroll
            for (int k = 0; k < 7; ++k) c3[k] = renorm(fmadd_u(f[k], t[k], c3[k]));
            more[kE5] = add_u(more[kE5], me5);
            const T w[5] = {g.xx, g.yy, g.xy2, g.xz2, g.yz2};
#pragma unroll
            for (int k = 0; k < 5; ++k) more[kC7 + k] = fmadd_u(me7, w[k], more[kC7 + k]);
            const T me9 = mul_u(m, g.e9);
            const T hx = mul_u(me9, g.xx), hy = mul_u(me9, g.yy);
            T *c4 = more + kC4;
            c4[0] = fmadd_u(hx, g.xx, c4[0]);
            c4[1] = fmadd_u(hx, g.xy2, c4[1]);
            c4[2] = fmadd_u(hx, g.xz2, c4[2]);
            c4[3] = fmadd_u(hx, g.yy, c4[3]);
            c4[4] = fmadd_u(hx, g.yz2, c4[4]);
            c4[5] = fmadd_u(hy, g.xy2, c4[5]);
            c4[6] = fmadd_u(hy, g.xz2, c4[6]);
            c4[7] = fmadd_u(hy, g.yy, c4[7]);
            c4[8] = fmadd_u(hy, g.yz2, c4[8]);
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) more[kV + k] = fmadd_u(me5, g.R[k], more[kV + k]);
            const T f[7] = {gx, gy, gx, gx, gx, gy, gy}, t[7] = {g.xx, g.xx, g.xz2, g.yy, g.yz2, g.yy, g.yz2};
#pragma unroll
            for (int k = 0; k < 7; ++k) c3[k] = fmadd_u(f[k], t[k], c3[k]);
        }
        low.add(g, me3, m, src, mp);
    }

    // the target's 16 traceless values (L0 | L1 | L2 xx yy xy xz yz | L3 xxx
    // xxy xxz xyy xyz yyy yyz) and the correction.  own: the target's packed
    // data (its third, at order 2 second, moment over its mass enters the
    // correction).
    __device__ __forceinline__ void finish(const WideSrc<T> &own, T L[16], T S[3]) const
    {
        L[0] = -low.a0;
#pragma unroll
        for (int i = 0; i < 3; ++i) L[1 + i] = low.a1[i];
        L[4] = -c2[0];
        L[5] = -c2[1];
#pragma unroll
        for (int k = 2; k < 5; ++k) L[4 + k] = scaled(-1.5f, c2[k]);
        low.correction(S);
        if constexpr (ORDER == 3) {
#pragma unroll
            for (int k = 0; k < 7; ++k) L[9 + k] = scaled(k == 4 ? 7.5f : 3.f, c3[k]);
            const T e5 = more[kE5], *c7 = more + kC7, *c4 = more + kC4;
            // S_i -= 7 C4_ijkl a_jkl - 3 C7_kl a_ikl, a = t3 / M0 of the target;
            // the zz components of the sums follow from r^2 e_k = e_(k-2)
            T a[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) a[k] = own.t3[k] / own.m0;
            const T axzz = -(a[0] + a[3]), ayzz = -(a[1] + a[5]), azzz = -(a[2] + a[6]);
            const T xxxx = c4[0], xxyy = c4[3], yyyy = c4[7];
            const T xxxy = scaled(0.5f, c4[1]), xxxz = scaled(0.5f, c4[2]), xxyz = scaled(0.5f, c4[4]);
            const T xyyy = scaled(0.5f, c4[5]), xyyz = scaled(0.5f, c4[6]), yyyz = scaled(0.5f, c4[8]);
            const T xx = c7[0], yy = c7[1], zz = e5 - xx - yy;
            const T xy = scaled(0.5f, c7[2]), xz = scaled(0.5f, c7[3]), yz = scaled(0.5f, c7[4]);
            const T xxzz = xx - xxxx - xxyy, xyzz = xy - xxxy - xyyy, xzzz = xz - xxxz - xyyz;
            const T yyzz = yy - xxyy - yyyy, yzzz = yz - xxyz - yyyz, zzzz = zz - xxzz - yyzz;
            const T C4[3][10] = {{xxxx, xxxy, xxxz, xxyy, xxyz, xxzz, xyyy, xyyz, xyzz, xzzz},
                                 {xxxy, xxyy, xxyz, xyyy, xyyz, xyzz, yyyy, yyyz, yyzz, yzzz},
                                 {xxxz, xxyz, xxzz, xyyz, xyzz, xzzz, yyyz, yyzz, yzzz, zzzz}};
            const T w3[10] = {a[0], a[1], a[2], a[3], a[4], axzz, a[5], a[6], ayzz, azzz};
            const T C7[6] = {xx, xy, xz, yy, yz, zz};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                T p = T(0), r = T(0);
#pragma unroll
                for (int k = 0; k < 10; ++k) p = fmadd(scaled(float(mult3(k)), w3[k]), C4[i][k], p);
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    r = fmadd(scaled(float(mult2(k)), w3[r3_of(i, k)]), C7[k], r);
                S[i] = S[i] - (scaled(7.f, p) - scaled(3.f, r));
            }
        } else {
#pragma unroll
            for (int k = 9; k < 16; ++k) L[k] = T(0);
            // S_i += 5 C3_ijk a_jk - 2 V_j a_ij, a = t2 / M0 of the target
            T a[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) a[k] = own.t2[k] / own.m0;
            const T azz = -(a[0] + a[1]);
            const T *v = more + kV;
            const T xxx = c3[0], xxy = c3[1], xyy = c3[3], yyy = c3[5];
            const T xxz = scaled(0.5f, c3[2]), xyz = scaled(0.5f, c3[4]), yyz = scaled(0.5f, c3[6]);
            const T C3[10] = {xxx, xxy, xxz, xyy, xyz, v[0] - xxx - xyy, yyy, yyz, v[1] - xxy - yyy,
                              v[2] - xxz - yyz};
            const T w2[6] = {a[0], a[2], a[3], a[1], a[4], azz};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                T p = T(0), r = T(0);
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    p = fmadd(scaled(float(mult2(k)), w2[k]), C3[r3_of(i, k)], p);
#pragma unroll
                for (int j = 0; j < 3; ++j) r = fmadd(w2[r2_of(i, j)], v[j], r);
                S[i] = S[i] + (scaled(5.f, p) - scaled(2.f, r));
            }
        }
    }
};

// A target's sums over the stencil, in chunks of 16 entries.  double: the
// chunk's sums are added to the totals and start again at zero (one long sum
// drifts: neighbouring sources contribute nearly equal terms, whose roundings
// agree in sign; 3e-15 instead of 4e-16 of L0 on the workloads).  double-float:
// the running sums are put back into canonical form (they take unnormalised
// terms).
template <typename T, class Sums>
struct WideChunked {
    Sums part, sum;
    __device__ __forceinline__ void zero()
    {
        part.zero();
        sum.zero();
    }
    __device__ __forceinline__ void flush()
    {
        T *p = reinterpret_cast<T *>(&part), *t = reinterpret_cast<T *>(&sum);
#pragma unroll
        for (int k = 0; k < int(sizeof(Sums) / sizeof(T)); ++k) t[k] += p[k];
        part.zero();
    }
    __device__ __forceinline__ Sums &total() { return sum; }
};
template <class Sums>
struct WideChunked<dfloat, Sums> {
    Sums part;
    __device__ __forceinline__ void zero() { part.zero(); }
    __device__ __forceinline__ void flush() { part.flush(); }
    __device__ __forceinline__ Sums &total() { return part; }
};

// a refined source into a leaf target
template <typename T, int ORDER>
__device__ __forceinline__ void wide_add_leaf(T x, T y, T z, const WideSrc<T> &src, WideLow<T, ORDER> &A)
{
    WideGeo<T> g;
    g.template eval<ORDER>(x, y, z);
    A.add(g, product(src.m0, g.e3), src.m0, src, true);
}

}  // namespace fmm
