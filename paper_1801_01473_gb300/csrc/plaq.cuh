// plaq.cuh -- what the plaquette-sharing link kernels have in common: the geometry of a site's
// plaquettes, matrices held as structure-of-arrays workspaces, anti-Hermitian and Hermitian 3x3
// matrices by their 9 real numbers, and exp(iQ) of a Hermitian Q in that form.
//
// For an ordered pair of directions (mu, nu) and a site x,
//   P(mu, nu)(x)   = U_nu(x) U_mu(x+nu)             the corner path x -> x+nu -> x+nu+mu
//   Sup(mu, nu)(x) = P(mu, nu)(x) U_nu(x+mu)^dag    the upper staple of link (x, mu)
//   Slo(mu, nu)(x) = U_nu(x)^dag P(nu, mu)(x)       the lower staple of link (x+nu, mu)
// Each is one product, made once per plaquette instead of once per link that uses it.  FP64
// kernels on GB300 are bound by the FP64 pipe (2 multiply-adds per clock and SM, ~0.58e12/s), so
// the number of 3x3 products decides their time and the extra memory traffic does not show.
#pragma once

#include "su3.cuh"

namespace stg {
namespace plaq {
using namespace su3;

struct PlaqGeo {
    int L[4], stride[4];
    int V;
    FastDiv by_stride[4], by_L[4];
};

inline PlaqGeo plaq_geo(const Geom &geo)
{
    PlaqGeo g;
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

__device__ __forceinline__ int coord(const PlaqGeo &g, int i, int mu)
{
    const int q = fast_div(i, g.by_stride[mu]);
    return q - fast_div(q, g.by_L[mu]) * g.L[mu];
}

// neighbours of site i along mu (periodic)
__device__ __forceinline__ int up(const PlaqGeo &g, int i, int mu)
{
    return coord(g, i, mu) == g.L[mu] - 1 ? i - (g.L[mu] - 1) * g.stride[mu] : i + g.stride[mu];
}
__device__ __forceinline__ int down(const PlaqGeo &g, int i, int mu)
{
    return coord(g, i, mu) == 0 ? i + (g.L[mu] - 1) * g.stride[mu] : i - g.stride[mu];
}

// The 6 planes (m < n) in the order 01 02 03 12 13 23; an ordered pair (mu, nu) is slot 2 p of its
// plane p when mu < nu and slot 2 p + 1 otherwise.
__host__ __device__ __forceinline__ int plane_of(int mu, int nu)
{
    const int m = mu < nu ? mu : nu, n = mu < nu ? nu : mu;
    return m * (7 - m) / 2 + n - m - 1;
}
__device__ __forceinline__ int slot_of(int mu, int nu) { return 2 * plane_of(mu, nu) + (mu > nu ? 1 : 0); }
__device__ __forceinline__ void plane_dirs(int p, int &m, int &n)
{
    m = p < 3 ? 0 : p < 5 ? 1 : 2;
    n = p < 3 ? p + 1 : p < 5 ? p - 1 : 3;
}

// matrix of canonical links [4][V][3][3]
template <typename T>
__device__ __forceinline__ M3T<T> link_at(const typename C2<T>::type *__restrict__ U, const PlaqGeo &g, int mu, int i)
{
    M3T<T> a;
    const typename C2<T>::type *p = U + ((long long)mu * g.V + i) * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const typename C2<T>::type v = p[k];
        a.m[k / 3][k % 3] = cx<T>{v.x, v.y};
    }
    return a;
}

// Workspace of matrices, structure of arrays: field f holds [9][V] complex numbers, so a warp's
// accesses are contiguous.
template <typename T>
__device__ __forceinline__ M3T<T> ws_ld(const typename C2<T>::type *__restrict__ base, int V, int f, int i)
{
    M3T<T> a;
    const typename C2<T>::type *p = base + (long long)f * 9 * V + i;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const typename C2<T>::type v = p[(long long)k * V];
        a.m[k / 3][k % 3] = cx<T>{v.x, v.y};
    }
    return a;
}
template <typename T>
__device__ __forceinline__ void ws_st(typename C2<T>::type *__restrict__ base, int V, int f, int i, const M3T<T> &a)
{
    typename C2<T>::type *p = base + (long long)f * 9 * V + i;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        typename C2<T>::type v;
        v.x = a.m[k / 3][k % 3].re;
        v.y = a.m[k / 3][k % 3].im;
        p[(long long)k * V] = v;
    }
}

// acc += w a
template <typename T>
__device__ __forceinline__ void axpy3(M3T<T> &acc, T w, const M3T<T> &a)
{
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            acc.m[r][c].re = fma(w, a.m[r][c].re, acc.m[r][c].re);
            acc.m[r][c].im = fma(w, a.m[r][c].im, acc.m[r][c].im);
        }
}

// ------------------------------------------------------------------ 9-number matrices
// H9 d, o: Hermitian (diagonal d, upper triangle o = 01, 02, 12, lower triangle its conjugate) or
// anti-Hermitian (diagonal i d, upper triangle o, lower triangle -conj(o)).
template <typename T>
struct H9 {
    T d[3];
    cx<T> o[3];
};

// anti-Hermitian part (Z - Z^dag)/2 of Z = op(a) op(b): 90 multiply-adds instead of a product's 108
template <bool DA, bool DB, typename T>
__device__ __forceinline__ H9<T> anti_mul(const M3T<T> &a, const M3T<T> &b)
{
    H9<T> z;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        T s = T(0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const cx<T> x = el<DA>(a, r, k), y = el<DB>(b, k, r);
            s = fma(x.re, y.im, s);
            s = fma(x.im, y.re, s);
        }
        z.d[r] = s;
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int r = e == 2 ? 1 : 0, c = e == 0 ? 1 : 2;
        T re = T(0), im = T(0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            cx<T> x = el<DA>(a, r, k), y = el<DB>(b, k, c);
            re = fma(x.re, y.re, re);
            re = fma(-x.im, y.im, re);
            im = fma(x.re, y.im, im);
            im = fma(x.im, y.re, im);
            x = el<DA>(a, c, k), y = el<DB>(b, k, r);
            re = fma(-x.re, y.re, re);
            re = fma(x.im, y.im, re);
            im = fma(x.re, y.im, im);
            im = fma(x.im, y.re, im);
        }
        z.o[e] = cx<T>{T(0.5) * re, T(0.5) * im};
    }
    return z;
}

// the full matrix of a traceless anti-Hermitian part: diagonal i (d - tr/3)
template <typename T>
__device__ __forceinline__ M3T<T> expand_anti_traceless(const H9<T> &z)
{
    const T tr = (z.d[0] + z.d[1] + z.d[2]) / T(3);
    M3T<T> y;
#pragma unroll
    for (int r = 0; r < 3; ++r) y.m[r][r] = cx<T>{T(0), z.d[r] - tr};
    y.m[0][1] = z.o[0];
    y.m[0][2] = z.o[1];
    y.m[1][2] = z.o[2];
    y.m[1][0] = cx<T>{-z.o[0].re, z.o[0].im};
    y.m[2][0] = cx<T>{-z.o[1].re, z.o[1].im};
    y.m[2][1] = cx<T>{-z.o[2].re, z.o[2].im};
    return y;
}

}  // namespace plaq
}  // namespace stg
