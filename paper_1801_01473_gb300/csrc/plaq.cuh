// plaq.cuh -- what the plaquette-sharing link kernels have in common: the planes of a site, matrices
// held as structure-of-arrays workspaces, anti-Hermitian and Hermitian 3x3 matrices by their 9 real
// numbers.
//
// For an ordered pair of directions (mu, nu) and a site x,
//   P(mu, nu)(x)   = U_nu(x) U_mu(x+nu)             the corner path x -> x+nu -> x+nu+mu
//   Sup(mu, nu)(x) = P(mu, nu)(x) U_nu(x+mu)^dag    the upper staple of link (x, mu)
//   Slo(mu, nu)(x) = U_nu(x)^dag P(nu, mu)(x)       the lower staple of link (x+nu, mu)
// Each is one product, made once per plaquette instead of once per link that uses it.  FP64
// kernels on GB300 are bound by the FP64 pipe (2 multiply-adds per clock and SM, ~0.58e12/s), so
// the number of 3x3 products decides their time and the extra memory traffic does not show.
#pragma once

#include "dslash.cuh"  // launch_overlap
#include "stg_common.h"
#include "su3.cuh"

namespace stg {
namespace plaq {
using namespace su3;

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
__device__ __forceinline__ M3T<T> link_at(const typename C2<T>::type *__restrict__ U, const LinkGeo &g, int mu, int i)
{
    M3T<T> a;
    ld(U, g, mu, i, a);
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

// link (mu, i) of canonical links or of a workspace of 4 fields
template <bool WS, typename T>
__device__ __forceinline__ M3T<T> link_of(const typename C2<T>::type *__restrict__ U, const LinkGeo &g, int mu, int i)
{
    if constexpr (WS) return ws_ld<T>(U, g.V, mu, i);
    return link_at<T>(U, g, mu, i);
}

// Canonical links -> workspace of 4 fields, through shared memory so that both sides are contiguous.
// A thread's 9 loads of a canonical FP32 link are 72 bytes apart between lanes and touch 18 lines
// per instruction where the workspace's touch 2; the FP32 link kernels were bound by that.
constexpr int kWsTile = 128;
template <typename T>
__global__ void __launch_bounds__(kWsTile) k_links_to_ws(const typename C2<T>::type *__restrict__ src,
                                                         typename C2<T>::type *__restrict__ dst, int V)
{
    using C = typename C2<T>::type;
    pdl_enter();
    __shared__ C tile[kWsTile * 9];
    const int i0 = blockIdx.x * kWsTile, n = min(kWsTile, V - i0), mu = blockIdx.y;
    const C *s = src + ((long long)mu * V + i0) * 9;
    for (int k = threadIdx.x; k < n * 9; k += kWsTile) tile[k] = s[k];
    __syncthreads();
    if ((int)threadIdx.x < n)
#pragma unroll
        for (int k = 0; k < 9; ++k) dst[((long long)mu * 9 + k) * V + i0 + threadIdx.x] = tile[threadIdx.x * 9 + k];
}

// Whether the launches of a link operation may overlap (programmatic launch).  The blocks of the next kernel are
// then placed while the running one holds its SMs: they gather on the SMs that it leaves idle, or are
// stacked unevenly on top of it, and stay there.  That costs nothing while both kernels' warps find a quarter SM
// each (`pair` warps per 32 sites for two consecutive launches, `fits` per SM) and little from `large` sites
// up, where most blocks start later; between, plain launches are faster although each costs 2 to 3 us:
//   FP64, overlapping -> plain, back to back calls: chain rule 576 sites 264 -> 250 us, 1296 426 -> 250, 3072 552 -> 264,
//   6400 600 -> 473, 10000 731 -> 751; gauge force 256 sites 77 -> 83, 3072 169 -> 103, 6400 184 -> 162, 10000 275 ->
//   280; smearing 256 89 -> 97, 3072 189 -> 101, 10000 306 -> 289, 20736 500 -> 483, 32256 664 -> 674.
//   FP32 chain rule: 3072 44 -> 52, 4096 55 -> 50, 10000 78 -> 69, 20736 86 -> 93.
inline bool overlap(long long V, int pair, int fits, long long large)
{
    return pair * ((V + 31) / 32) <= (long long)fits * sm_count() || V >= large;
}

template <typename T>
cudaError_t links_to_ws(bool overlap, const void *links, typename C2<T>::type *ws, int V, cudaStream_t st)
{
    const dim3 tiles((unsigned)((V + kWsTile - 1) / kWsTile), 4);
    return launch_overlap(overlap, k_links_to_ws<T>, tiles, dim3(kWsTile), 0, st,
                          static_cast<const typename C2<T>::type *>(links), ws, V);
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

// Workspace of 9-number matrices: field f holds [9][V] reals (diagonal, then re, im of the triangle).
template <typename T>
__device__ __forceinline__ H9<T> ws_ld9(const T *__restrict__ base, int V, int f, int i)
{
    const T *p = base + (long long)f * 9 * V + i;
    T v[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = p[(long long)k * V];
    H9<T> z;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        z.d[k] = v[k];
        z.o[k] = cx<T>{v[3 + 2 * k], v[4 + 2 * k]};
    }
    return z;
}
template <typename T>
__device__ __forceinline__ void ws_st9(T *__restrict__ base, int V, int f, int i, const H9<T> &z)
{
    T *p = base + (long long)f * 9 * V + i;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[(long long)k * V] = z.d[k];
        p[(long long)(3 + 2 * k) * V] = z.o[k].re;
        p[(long long)(4 + 2 * k) * V] = z.o[k].im;
    }
}

// z += w a
template <typename T>
__device__ __forceinline__ void axpy9(H9<T> &z, T w, const H9<T> &a)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        z.d[k] = fma(w, a.d[k], z.d[k]);
        z.o[k].re = fma(w, a.o[k].re, z.o[k].re);
        z.o[k].im = fma(w, a.o[k].im, z.o[k].im);
    }
}

// acc += w b for an anti-Hermitian w (90 multiply-adds)
template <typename T>
__device__ __forceinline__ void anti_mul_acc(M3T<T> &acc, const H9<T> &w, const M3T<T> &b)
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            acc.m[r][c].re = fma(-w.d[r], b.m[r][c].im, acc.m[r][c].re);
            acc.m[r][c].im = fma(w.d[r], b.m[r][c].re, acc.m[r][c].im);
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int r = e == 2 ? 1 : 0, k = e == 0 ? 1 : 2;
            cmac(acc.m[r][c], w.o[e], b.m[k][c]);
            cmac_conj(acc.m[k][c], cx<T>{-w.o[e].re, -w.o[e].im}, b.m[r][c]);
        }
    }
}

// square of a Hermitian matrix
template <typename T>
__device__ __forceinline__ H9<T> square9(const H9<T> &q)
{
    const T n01 = q.o[0].re * q.o[0].re + q.o[0].im * q.o[0].im, n02 = q.o[1].re * q.o[1].re + q.o[1].im * q.o[1].im,
            n12 = q.o[2].re * q.o[2].re + q.o[2].im * q.o[2].im;
    H9<T> s;
    s.d[0] = fma(q.d[0], q.d[0], n01 + n02);
    s.d[1] = fma(q.d[1], q.d[1], n01 + n12);
    s.d[2] = fma(q.d[2], q.d[2], n02 + n12);
    const T t01 = q.d[0] + q.d[1], t02 = q.d[0] + q.d[2], t12 = q.d[1] + q.d[2];
    s.o[0] = cx<T>{t01 * q.o[0].re, t01 * q.o[0].im};
    cmac_conj(s.o[0], q.o[2], q.o[1]);  // q02 conj(q12)
    s.o[1] = cx<T>{t02 * q.o[1].re, t02 * q.o[1].im};
    cmac(s.o[1], q.o[0], q.o[2]);
    s.o[2] = cx<T>{t12 * q.o[2].re, t12 * q.o[2].im};
    cmac_conj(s.o[2], q.o[0], q.o[1]);  // conj(q01) q02
    return s;
}

// q n + n q of two Hermitian matrices
template <typename T>
__device__ __forceinline__ H9<T> anticommutator9(const H9<T> &q, const H9<T> &n)
{
    T p[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = fma(q.o[k].re, n.o[k].re, q.o[k].im * n.o[k].im);
    H9<T> s;
    s.d[0] = T(2) * fma(q.d[0], n.d[0], p[0] + p[1]);
    s.d[1] = T(2) * fma(q.d[1], n.d[1], p[0] + p[2]);
    s.d[2] = T(2) * fma(q.d[2], n.d[2], p[1] + p[2]);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int r = e == 2 ? 1 : 0, c = e == 0 ? 1 : 2;
        const T tq = q.d[r] + q.d[c], tn = n.d[r] + n.d[c];
        s.o[e].re = fma(tq, n.o[e].re, tn * q.o[e].re);
        s.o[e].im = fma(tq, n.o[e].im, tn * q.o[e].im);
    }
    cmac_conj(s.o[0], n.o[2], q.o[1]);  // q02 conj(n12)
    cmac_conj(s.o[0], q.o[2], n.o[1]);  // n02 conj(q12)
    cmac(s.o[1], q.o[0], n.o[2]);
    cmac(s.o[1], n.o[0], q.o[2]);
    cmac_conj(s.o[2], q.o[0], n.o[1]);
    cmac_conj(s.o[2], n.o[0], q.o[1]);
    return s;
}

// c0 = det q and c1 = tr q^2 / 2 of a Hermitian q with square q2
template <typename T>
__device__ __forceinline__ void char_coefs9(const H9<T> &q, const H9<T> &q2, T &c0, T &c1)
{
    c1 = T(0.5) * (q2.d[0] + q2.d[1] + q2.d[2]);
    // det q = Re of the expansion along the first row, q10 = conj(q01) and so on
    const T n01 = q.o[0].re * q.o[0].re + q.o[0].im * q.o[0].im, n02 = q.o[1].re * q.o[1].re + q.o[1].im * q.o[1].im,
            n12 = q.o[2].re * q.o[2].re + q.o[2].im * q.o[2].im;
    const cx<T> t = cmul(q.o[0], q.o[2]);  // q01 q12, to be taken with q20 = conj(q02)
    const T re = fma(t.re, q.o[1].re, t.im * q.o[1].im);
    c0 = fma(q.d[0], fma(q.d[1], q.d[2], -n12), fma(T(2), re, -fma(q.d[1], n02, q.d[2] * n01)));
}

// f0 + f1 q + f2 q2 of Hermitian q, q2
template <typename T>
__device__ __forceinline__ M3T<T> poly9(const cx<T> f[3], const H9<T> &q, const H9<T> &q2)
{
    M3T<T> e;
#pragma unroll
    for (int r = 0; r < 3; ++r)
        e.m[r][r] = cx<T>{fma(f[1].re, q.d[r], fma(f[2].re, q2.d[r], f[0].re)),
                          fma(f[1].im, q.d[r], fma(f[2].im, q2.d[r], f[0].im))};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int r = k == 2 ? 1 : 0, c = k == 0 ? 1 : 2;
        cx<T> v = cmul(f[1], q.o[k]);
        cmac(v, f[2], q2.o[k]);
        e.m[r][c] = v;
        v = cmul(f[1], cconj(q.o[k]));
        cmac(v, f[2], cconj(q2.o[k]));
        e.m[c][r] = v;
    }
    return e;
}

}  // namespace plaq
}  // namespace stg
