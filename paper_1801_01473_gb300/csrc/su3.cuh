// su3.cuh -- 3x3 complex matrices in registers (T = double or float), for the kernels that work on
// whole links in the canonical layout [4][V][3][3] (complex128, or complex64 for the FP32 variants
// of the MD kernels): loads/stores, products with optional daggers, the traceless anti-Hermitian
// projection, lexicographic neighbours, and exp(iQ) of a traceless Hermitian Q as
// f0 + f1 Q + f2 Q^2 (with the derivatives of the f_j for chain rules).
#pragma once

#include "stg_internal.cuh"

namespace stg {
namespace su3 {

template <typename T>
struct M3T {
    cx<T> m[3][3];
};
using M3 = M3T<double>;

// storage type of one complex number of precision T
template <typename T>
struct C2;
template <>
struct C2<double> {
    using type = double2;
};
template <>
struct C2<float> {
    using type = float2;
};

struct LinkGeo {
    int L[4], stride[4];
    int V;
    FastDiv by_stride[4], by_L[4];
};

// Site numbers are 32 bits: 2^31 sites, which a lattice may have, are refused by the link operations (their
// FP32 links alone would take 618 GB).
constexpr long long kMaxLinkSites = 0x7fffffffLL;

inline LinkGeo link_geo(const Geom &geo)
{
    LinkGeo g;
    long long s = 1;
    for (int mu = 0; mu < 4; ++mu) {
        g.L[mu] = geo.L[mu];
        g.stride[mu] = (int)s;
        g.by_stride[mu] = make_fast_div((unsigned)s);
        g.by_L[mu] = make_fast_div((unsigned)geo.L[mu]);
        s *= geo.L[mu];
    }
    g.V = (int)s;
    return g;
}

// coordinate mu of site i
__device__ __forceinline__ int coord(const LinkGeo &g, int i, int mu)
{
    const int q = fast_div(i, g.by_stride[mu]);
    return q - fast_div(q, g.by_L[mu]) * g.L[mu];
}

// neighbours of site i along mu (periodic)
__device__ __forceinline__ int up(const LinkGeo &g, int i, int mu)
{
    return coord(g, i, mu) == g.L[mu] - 1 ? i - (g.L[mu] - 1) * g.stride[mu] : i + g.stride[mu];
}
__device__ __forceinline__ int down(const LinkGeo &g, int i, int mu)
{
    return coord(g, i, mu) == 0 ? i + (g.L[mu] - 1) * g.stride[mu] : i - g.stride[mu];
}

template <typename T>
__device__ __forceinline__ void ld(const typename C2<T>::type *__restrict__ base, const LinkGeo &g, int mu, int i,
                                   M3T<T> &a)
{
    const typename C2<T>::type *p = base + ((long long)mu * g.V + i) * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const typename C2<T>::type v = p[k];
        a.m[k / 3][k % 3] = cx<T>{v.x, v.y};
    }
}

template <typename T>
__device__ __forceinline__ void st(typename C2<T>::type *__restrict__ base, const LinkGeo &g, int mu, int i,
                                   const M3T<T> &a)
{
    typename C2<T>::type *p = base + ((long long)mu * g.V + i) * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        p[k].x = a.m[k / 3][k % 3].re;
        p[k].y = a.m[k / 3][k % 3].im;
    }
}

// element (r, c) of a or of a^dag
template <bool D, typename T>
__device__ __forceinline__ cx<T> el(const M3T<T> &a, int r, int c)
{
    return D ? cconj(a.m[c][r]) : a.m[r][c];
}

// acc (+)= op(a) op(b)
template <bool DA, bool DB, typename T>
__device__ __forceinline__ void mul_acc(M3T<T> &acc, const M3T<T> &a, const M3T<T> &b)
{
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < 3; ++k) cmac(acc.m[r][c], el<DA>(a, r, k), el<DB>(b, k, c));
}

template <typename T = double>
__device__ __forceinline__ M3T<T> zero3()
{
    M3T<T> z;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) z.m[r][c] = cx<T>{T(0), T(0)};
    return z;
}

template <bool DA, bool DB, typename T>
__device__ __forceinline__ M3T<T> mul(const M3T<T> &a, const M3T<T> &b)
{
    M3T<T> z = zero3<T>();
    mul_acc<DA, DB>(z, a, b);
    return z;
}

// TA(X) = (X - X^dag)/2 - tr(X - X^dag)/6
template <typename T>
__device__ __forceinline__ M3T<T> ta(const M3T<T> &x)
{
    M3T<T> y;
    const T im_tr = (x.m[0][0].im + x.m[1][1].im + x.m[2][2].im) / T(3);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            y.m[r][c] = cx<T>{T(0.5) * (x.m[r][c].re - x.m[c][r].re), T(0.5) * (x.m[r][c].im + x.m[c][r].im)};
            if (r == c) y.m[r][c].im -= im_tr;
        }
    return y;
}

// f_j of exp(iQ) = f0 + f1 Q + f2 Q^2 and (DERIV) df_j/dc0, df_j/dc1.
template <typename T>
struct ExpCoefT {
    cx<T> f[3], d0[3], d1[3];
};
using ExpCoef = ExpCoefT<double>;

// 1/n!, n = 0..131
template <typename T>
struct InvFactorial {
    T v[132];
    constexpr InvFactorial() : v{}
    {
        double f = 1.0;
        for (int n = 0; n < 132; ++n) {
            v[n] = f < (sizeof(T) == 4 ? 1e-37 : 0.0) ? T(0) : (T)f;
            f /= n + 1;
        }
    }
};
__constant__ constexpr InvFactorial<double> kInvFactorial64{};
__constant__ constexpr InvFactorial<float> kInvFactorial32{};
template <typename T>
__device__ __forceinline__ T inv_factorial(int n)
{
    return sizeof(T) == 8 ? (T)kInvFactorial64.v[n] : (T)kInvFactorial32.v[n];
}

// exp(iQ) = f0 + f1 Q + f2 Q^2 with (DERIV) the derivatives of the f_j, from one sequence.
// Q^3 = c1 Q + c0 gives Q^n = c0 h_{n-1} + h_{n+1} Q + h_n Q^2 (n >= 1) with
//   h_0 = h_1 = 0, h_2 = 1, h_{n+1} = c1 h_{n-1} + c0 h_{n-2},
// and g_n = dh_n/dc0 satisfies dh_n/dc1 = g_{n+1} (both from the generating function
// t^2 / (1 - c1 t^2 - c0 t^3)), g_{n+1} = c1 g_{n-1} + c0 g_{n-2} + h_{n-2}.  So with s_n = i^n / n!
//   f2 = sum s_n h_n, f1 = sum s_n h_{n+1}, f0 = 1 + c0 sum s_n h_{n-1},
//   df2/dc0 = sum s_n g_n,  df2/dc1 = df1/dc0 = sum s_n g_{n+1},  df1/dc1 = sum s_n g_{n+2},
//   df0/dc0 = sum s_n h_{n-1} + c0 sum s_n g_{n-1},  df0/dc1 = c0 df2/dc0:
// 5 (12 with derivatives) multiply-adds per term, no divisions.  The number of terms is settled
// beforehand in FP32: the rest of the coefficients, and of their derivatives (polynomial in n times
// r^n/n!, r >= the spectral radius of Q), lies below the precision's resolution.
template <bool DERIV, typename T>
__device__ __forceinline__ ExpCoefT<T> exp_sums(T c0, T c1)
{
    int nmax = 6;
    {
        const float stop = sizeof(T) == 4 ? 1e-9f : 1e-18f;
        float r = sqrtf(fmaxf(2.f * (float)c1, 0.f));
        if (!(r >= 1.f)) r = 1.f;
        float bound = 1.f;  // r^n / n!
        for (int n = 1; n < 128; ++n) {
            bound *= __fdividef(r, (float)n);
            const float m = (float)(n + 1);
            nmax = n;
            if (n >= 6 && bound * m * m * m < stop) break;
        }
    }
    T hm = T(0), h = T(0), hp = T(1);               // h_{n-1}, h_n, h_{n+1} at n = 1
    T gm = T(0), g = T(0), gp = T(0), gpp = T(0);               // g_{n-1}, g_n, g_{n+1}, g_{n+2}
    T s0[2] = {T(0), T(0)}, s1[2] = {T(0), T(0)}, s2[2] = {T(0), T(0)};  // sums of h_{n-1}, h_n, h_{n+1}; [1] odd n
    T d0[2] = {T(0), T(0)}, d1[2] = {T(0), T(0)}, d2[2] = {T(0), T(0)}, d3[2] = {T(0), T(0)};  // g_{n-1} .. g_{n+2}
#pragma unroll 1
    for (int n0 = 1; n0 <= nmax; n0 += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {  // n = n0 + u = 1 + u mod 4: i^n = i, -1, -i, 1
            T s = inv_factorial<T>(n0 + u);
            if (u == 1 || u == 2) s = -s;
            const int o = (u & 1) ? 0 : 1;
            s0[o] = fma(s, hm, s0[o]);
            s1[o] = fma(s, h, s1[o]);
            s2[o] = fma(s, hp, s2[o]);
            if (DERIV) {
                d0[o] = fma(s, gm, d0[o]);
                d1[o] = fma(s, g, d1[o]);
                d2[o] = fma(s, gp, d2[o]);
                d3[o] = fma(s, gpp, d3[o]);
                const T gn = fma(c1, gp, fma(c0, g, h));  // g_{n+3}
                gm = g; g = gp; gp = gpp; gpp = gn;
            }
            const T hn = fma(c1, h, c0 * hm);  // h_{n+2}
            hm = h; h = hp; hp = hn;
        }
    }
    ExpCoefT<T> e;
    e.f[0] = cx<T>{fma(c0, s0[0], T(1)), c0 * s0[1]};
    e.f[1] = cx<T>{s2[0], s2[1]};
    e.f[2] = cx<T>{s1[0], s1[1]};
    if (DERIV) {
        e.d0[0] = cx<T>{fma(c0, d0[0], s0[0]), fma(c0, d0[1], s0[1])};
        e.d0[1] = cx<T>{d2[0], d2[1]};
        e.d0[2] = cx<T>{d1[0], d1[1]};
        e.d1[0] = cx<T>{c0 * d1[0], c0 * d1[1]};
        e.d1[1] = cx<T>{d3[0], d3[1]};
        e.d1[2] = cx<T>{d2[0], d2[1]};
    }
    return e;
}

// c0 = det Q, c1 = tr Q^2 / 2 of a Hermitian Q (both real)
template <typename T>
__device__ __forceinline__ void char_coefs(const M3T<T> &q, const M3T<T> &q2, T &c0, T &c1)
{
    c1 = T(0.5) * (q2.m[0][0].re + q2.m[1][1].re + q2.m[2][2].re);
    // det = q00 (q11 q22 - q12 q21) - q01 (q10 q22 - q12 q20) + q02 (q10 q21 - q11 q20)
    cx<T> t = cmul(q.m[1][1], q.m[2][2]), u = cmul(q.m[1][2], q.m[2][1]);
    const cx<T> d = cmul(q.m[0][0], cx<T>{t.re - u.re, t.im - u.im});
    t = cmul(q.m[1][0], q.m[2][2]); u = cmul(q.m[1][2], q.m[2][0]);
    const cx<T> e1 = cmul(q.m[0][1], cx<T>{t.re - u.re, t.im - u.im});
    t = cmul(q.m[1][0], q.m[2][1]); u = cmul(q.m[1][1], q.m[2][0]);
    const cx<T> e2 = cmul(q.m[0][2], cx<T>{t.re - u.re, t.im - u.im});
    c0 = d.re - e1.re + e2.re;
}

// E = f0 + f1 Q + f2 Q^2
template <typename T>
__device__ __forceinline__ M3T<T> poly3(const cx<T> f[3], const M3T<T> &q, const M3T<T> &q2)
{
    M3T<T> e;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            cx<T> v = cmul(f[1], q.m[r][c]);
            cmac(v, f[2], q2.m[r][c]);
            if (r == c) { v.re += f[0].re; v.im += f[0].im; }
            e.m[r][c] = v;
        }
    return e;
}

}  // namespace su3
}  // namespace stg
