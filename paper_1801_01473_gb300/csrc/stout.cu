// stout.cu -- stout smearing of the gauge links and the force chain rule through it (Sec. 2:
// the Dirac operator uses the k-times stout-smeared links U^(k); Sec. 3: the MD evolves U^(0),
// so the fermion force is pulled back through the k smearing steps).
//
// One step, per link (x, mu):  C = rho * (sum of the six staples around the link),
// i Q = TA(C U^dag), U' = exp(iQ) U.  exp(iQ) = f0 + f1 Q + f2 Q^2: Q^n reduces to
// a_n + b_n Q + c_n Q^2 by the Cayley-Hamilton identity Q^3 = c1 Q + c0 (c0 = det Q,
// c1 = tr Q^2 / 2, Q traceless Hermitian), so the f_j are the Taylor series of exp with
// scalar coefficient recursions -- no transcendental functions, and entire in (c0, c1), so the
// chain rule needs no special case at degenerate eigenvalues.  The recursion also carries
// d/dc0 and d/dc1 of the coefficients for the backward pass.
//
// Gradients follow torch's convention (G = dS/dRe U + i dS/dIm U, dS = Re tr(G^dag dU)).  The
// backward step is two kernels: k_stout_back_link (per link: the exp/TA/Omega part, writes the
// link's own gradient terms and Y = rho G_Omega U, the gradient of the unweighted staple sum)
// and k_stout_back_staples (per link: adds the product-rule terms of every staple of the other
// links' C that contains this link, gathered from Y -- each output is written by one thread).
//
// Layout: canonical complex128 or complex64 [4][V][3][3] (site index x + Lx (y + Ly (z + Lz t))); one
// thread per link.  FP64 steps mostly go by shared plaquettes (further down).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "dslash.cuh"
#include "plaq.cuh"
#include "stg_common.h"
#include "su3.cuh"

namespace stg {
namespace {
using namespace plaq;

// Weighted staple sum C_mu(x) = rho * sum_{nu != mu} (upper + lower staple).
template <typename T>
__device__ M3T<T> staple_sum(const typename C2<T>::type *__restrict__ U, const LinkGeo &g, int mu, int i,
                             T rho)
{
    M3T<T> c = zero3<T>();
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        M3T<T> a, b, t;
        // U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
        a = link_at<T>(U, g, nu, i);
        b = link_at<T>(U, g, mu, up(g, i, nu));
        t = mul<false, false>(a, b);
        a = link_at<T>(U, g, nu, up(g, i, mu));
        mul_acc<false, true>(c, t, a);
        // U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
        const int xm = down(g, i, nu);
        a = link_at<T>(U, g, nu, xm);
        b = link_at<T>(U, g, mu, xm);
        t = mul<true, false>(a, b);
        a = link_at<T>(U, g, nu, up(g, xm, mu));
        mul_acc<false, false>(c, t, a);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) c.m[r][k] = cx<T>{rho * c.m[r][k].re, rho * c.m[r][k].im};
    return c;
}

// Q = -i rho TA(Z) from the anti-Hermitian part of Z
template <typename T>
__device__ __forceinline__ H9<T> q_of(const H9<T> &z, T rho)
{
    const T tr = (z.d[0] + z.d[1] + z.d[2]) / T(3);
    H9<T> q;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        q.d[k] = rho * (z.d[k] - tr);
        q.o[k] = cx<T>{rho * z.o[k].im, -rho * z.o[k].re};
    }
    return q;
}

// One link of the chain rule: with G' = gp the gradient of the smeared link E U, E = exp(iQ), sets
// gu = E^dag G' and w = rho G_Omega, G_Omega = TA(i G_Q) the gradient of the algebra element.
template <typename T>
__device__ __forceinline__ void exp_gradient(const H9<T> &q, const M3T<T> &u, const M3T<T> &gp, T rho, M3T<T> &gu,
                                             H9<T> &w)
{
    const H9<T> q2 = square9(q);
    T c0, c1;
    char_coefs9(q, q2, c0, c1);
    const ExpCoefT<T> e = exp_sums<true>(c0, c1);
    gu = mul<true, false>(poly9(e.f, q, q2), gp);
    const M3T<T> M = mul<false, true>(gp, u);  // gradient of E
    // t_j = tr(M^dag Q^j);  K0, K1 = sum_j Re(t_j df_j/dc0,1)
    cx<T> t[3];
    t[0] = cx<T>{M.m[0][0].re + M.m[1][1].re + M.m[2][2].re, -(M.m[0][0].im + M.m[1][1].im + M.m[2][2].im)};
#pragma unroll
    for (int j = 1; j < 3; ++j) {
        const H9<T> &h = j == 1 ? q : q2;
        cx<T> s = cx<T>{T(0), T(0)};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            s.re = fma(M.m[r][r].re, h.d[r], s.re);
            s.im = fma(-M.m[r][r].im, h.d[r], s.im);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int r = k == 2 ? 1 : 0, c = k == 0 ? 1 : 2;
            cmac_conj(s, M.m[r][c], h.o[k]);
            cmac_conj(s, M.m[c][r], cconj(h.o[k]));
        }
        t[j] = s;
    }
    T K0 = T(0), K1 = T(0);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        K0 += t[j].re * e.d0[j].re - t[j].im * e.d0[j].im;
        K1 += t[j].re * e.d1[j].re - t[j].im * e.d1[j].im;
    }
    // Hermitian part of G_Q = K1 Q + K0 Q^2 + conj(f1) M + conj(f2) (M Q + Q M): the last term's is
    // the anticommutator of Q with the Hermitian part of conj(f2) M
    H9<T> n1, n2;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        n1.d[r] = fma(e.f[1].re, M.m[r][r].re, e.f[1].im * M.m[r][r].im);
        n2.d[r] = fma(e.f[2].re, M.m[r][r].re, e.f[2].im * M.m[r][r].im);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int r = k == 2 ? 1 : 0, c = k == 0 ? 1 : 2;
        const cx<T> s = M.m[r][c], z = cconj(M.m[c][r]);
        cx<T> v = cmul(cconj(e.f[1]), s);
        cmac(v, e.f[1], z);
        n1.o[k] = cx<T>{T(0.5) * v.re, T(0.5) * v.im};
        v = cmul(cconj(e.f[2]), s);
        cmac(v, e.f[2], z);
        n2.o[k] = cx<T>{T(0.5) * v.re, T(0.5) * v.im};
    }
    axpy9(n1, T(1), anticommutator9(q, n2));
    axpy9(n1, K1, q);
    axpy9(n1, K0, q2);
    // W = rho TA(i G_Q)
    const T tr = (n1.d[0] + n1.d[1] + n1.d[2]) / T(3);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        w.d[k] = rho * (n1.d[k] - tr);
        w.o[k] = cx<T>{-rho * n1.o[k].im, rho * n1.o[k].re};
    }
}

template <typename T>
struct StoutArgs {
    using C = typename C2<T>::type;
    LinkGeo g;
    T rho;
    const C *U;  // links of this step
    const C *Uws;  // their workspace copy (WS)
    const C *G;  // gradient of the step's output (backward)
    C *out;      // smeared links (forward) / gradient of U (backward)
    C *acc;      // the links' own gradient terms, between the backward kernels
    C *Y;        // rho G_Omega U (backward)
    int g_canon, out_canon, proj;  // G, out canonical; last step of kind 0: F = TA(U G^dag) instead of G
};

template <bool WS, typename T>
__device__ __forceinline__ void put(typename C2<T>::type *base, const LinkGeo &g, int mu, int i, const M3T<T> &a)
{
    if constexpr (WS)
        ws_st(base, g.V, mu, i, a);
    else
        st(base, g, mu, i, a);
}

constexpr int kStoutBlock = 128;

template <typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_fwd(const __grid_constant__ StoutArgs<T> a)
{
    pdl_enter();
    const int mu = threadIdx.x >> 5;  // warp-uniform
    const int i = blockIdx.x * 32 + (threadIdx.x & 31);
    if (i >= a.g.V) return;
    const M3T<T> u = link_at<T>(a.U, a.g, mu, i);
    const H9<T> q = q_of(anti_mul<false, true>(staple_sum<T>(a.U, a.g, mu, i, a.rho), u), T(1)), q2 = square9(q);
    T c0, c1;
    char_coefs9(q, q2, c0, c1);
    const ExpCoefT<T> e = exp_sums<false>(c0, c1);
    st(a.out, a.g, mu, i, mul<false, false>(poly9(e.f, q, q2), u));
}

template <bool WS, typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_back_link(const __grid_constant__ StoutArgs<T> a)
{
    pdl_enter();
    const int mu = threadIdx.x >> 5;  // warp-uniform
    const int i = blockIdx.x * 32 + (threadIdx.x & 31);
    if (i >= a.g.V) return;
    const M3T<T> C = staple_sum<T>(a.U, a.g, mu, i, a.rho);
    const M3T<T> u = link_at<T>(a.U, a.g, mu, i);
    M3T<T> gu;
    H9<T> go;
    const M3T<T> gp = WS && !a.g_canon ? ws_ld<T>(a.G, a.g.V, mu, i) : link_at<T>(a.G, a.g, mu, i);
    exp_gradient(q_of(anti_mul<false, true>(C, u), T(1)), u, gp, T(1), gu, go);
    M3T<T> y = zero3<T>();
    anti_mul_acc(y, go, u);
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) y.m[r][c] = cx<T>{a.rho * y.m[r][c].re, a.rho * y.m[r][c].im};
    put<WS>(a.Y, a.g, mu, i, y);
    // the link's own terms: E^dag G' + G_Omega^dag C
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        go.d[k] = -go.d[k];
        go.o[k] = cx<T>{-go.o[k].re, -go.o[k].im};
    }
    anti_mul_acc(gu, go, C);
    put<WS>(a.acc, a.g, mu, i, gu);
}

// Adds to the gradient of link (y, nu) the staple terms: for every mu != nu, the link sits in
//   C_mu(y)       as the first factor of the upper staple      -> Y_mu(y) U_nu(y+mu) U_mu(y+nu)^dag
//   C_mu(y+nu)    as the first factor of the lower staple      -> U_mu(y) U_nu(y+mu) Y_mu(y+nu)^dag
//   C_nu(y+mu)    as the middle factor of the lower staple     -> U_mu(y) Y_nu(y+mu) U_mu(y+nu)^dag
//   C_mu(y-mu)    as the last factor of the upper staple       -> Y_mu(y-mu)^dag U_nu(y-mu) U_mu(y-mu+nu)
//   C_mu(y-mu+nu) as the last factor of the lower staple       -> U_mu(y-mu)^dag U_nu(y-mu) Y_mu(y-mu+nu)
//   C_nu(y-mu)    as the middle factor of the upper staple     -> U_mu(y-mu)^dag Y_nu(y-mu) U_mu(y-mu+nu)
// with Y the gradient of the unweighted staple sums.
template <bool WS, typename T>
__global__ void __launch_bounds__(kStoutBlock, sizeof(T) == 4 ? 5 : 1) k_stout_back_staples(const __grid_constant__ StoutArgs<T> a)
{
    pdl_enter();
    const int nu = threadIdx.x >> 5;  // warp-uniform
    const int i = blockIdx.x * 32 + (threadIdx.x & 31);
    if (i >= a.g.V) return;
    const typename C2<T>::type *U = WS ? a.Uws : a.U;
    M3T<T> acc = link_of<WS, T>(a.acc, a.g, nu, i);
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
        if (mu == nu) continue;
        const int yp = up(a.g, i, mu), yn = up(a.g, i, nu);
        const int ym = down(a.g, i, mu), ymn = up(a.g, ym, nu);
        M3T<T> p, q, t;
        // forward side: U_nu(y+mu) shared by the first two terms
        p = link_of<WS, T>(U, a.g, nu, yp);   // U_nu(y+mu)
        q = link_of<WS, T>(U, a.g, mu, yn);   // U_mu(y+nu)
        t = mul<false, true>(p, q);
        q = link_of<WS, T>(a.Y, a.g, mu, i);    // Y_mu(y)
        mul_acc<false, false>(acc, q, t);
        q = link_of<WS, T>(U, a.g, mu, i);    // U_mu(y)
        t = mul<false, false>(q, p);
        p = link_of<WS, T>(a.Y, a.g, mu, yn);   // Y_mu(y+nu)
        mul_acc<false, true>(acc, t, p);
        p = link_of<WS, T>(a.Y, a.g, nu, yp);   // Y_nu(y+mu)
        t = mul<false, false>(q, p);
        q = link_of<WS, T>(U, a.g, mu, yn);   // U_mu(y+nu)
        mul_acc<false, true>(acc, t, q);
        // backward side: U_mu(y-mu)^dag leads the last two terms
        p = link_of<WS, T>(U, a.g, nu, ym);   // U_nu(y-mu)
        q = link_of<WS, T>(U, a.g, mu, ymn);  // U_mu(y-mu+nu)
        t = mul<false, false>(p, q);
        q = link_of<WS, T>(a.Y, a.g, mu, ym);   // Y_mu(y-mu)
        mul_acc<true, false>(acc, q, t);
        q = link_of<WS, T>(a.Y, a.g, mu, ymn);  // Y_mu(y-mu+nu)
        t = mul<false, false>(p, q);
        p = link_of<WS, T>(a.Y, a.g, nu, ym);   // Y_nu(y-mu)
        q = link_of<WS, T>(U, a.g, mu, ymn);  // U_mu(y-mu+nu)
        mul_acc<false, false>(t, p, q);
        p = link_of<WS, T>(U, a.g, mu, ym);   // U_mu(y-mu)
        mul_acc<true, false>(acc, p, t);
    }
    if (a.proj) acc = expand_anti_traceless(anti_mul<false, true>(link_of<WS, T>(U, a.g, nu, i), acc));
    if (WS && !a.out_canon)
        ws_st(a.out, a.g.V, nu, i, acc);
    else
        st(a.out, a.g, nu, i, acc);
}

// ------------------------------------------------------------------ by shared plaquettes
// The same step with every corner path made once per plaquette (plaq.cuh).  C U^dag is a sum over
// the plaquettes of the link of closed loops at its start: for the upper plaquette of (x, mu)
// P(mu, nu) P(nu, mu)^dag, whose anti-Hermitian part serves link (x, nu) with the opposite sign; for
// the lower one Slo(mu, nu)(x-nu) U_mu(x)^dag.  Only the anti-Hermitian parts are needed (9 numbers).
//
// Chain rule: with W = rho G_Omega of every link fixed, dS is the change of Re tr of the plaquettes
// when each link moves by Y = W U, so the gradient has the form of the rectangle force, with
//   P'(mu, nu)(x) = (W_nu - W_mu)(x) P(mu, nu)(x) + U_nu(x) Y_mu(x+nu)
//   G_mu(x) = E^dag G' + sum_nu [ P'(mu, nu)(x) U_nu(x+mu)^dag + P(mu, nu)(x) Y_nu(x+mu)^dag
//                               + U_nu(y)^dag P'(nu, mu)(y) ] - W_mu(x) sum_nu Slo(mu, nu)(y),  y = x - nu.
//
// ~1450 FP64 multiply-adds per link and smearing step (k_stout_fwd ~2300) and ~3700 per step of the
// chain rule (k_stout_back_* ~6850), both at the FP64 pipe's rate (0.58e12/s): two steps of 16^3x32
// 4.59 -> 2.65 ms, of the chain rule on 20x12x28x16 10.7 -> 5.7 ms.
template <typename T>
struct StoutPlaqArgs {
    using C = typename C2<T>::type;
    LinkGeo g;
    T rho;
    const C *U;    // links of this step
    const C *G;    // gradient of the step's output (backward)
    C *out;        // smeared links / gradient of U
    T *K, *Lo;     // anti-Hermitian loops: upper per plane [6], lower per ordered pair [12] (based at x)
    C *P, *Slo, *Pb;  // per ordered pair [12] (backward)
    T *W;          // [4] rho G_Omega, anti-Hermitian
    C *Y;          // [4] W U
    const C *proj;  // last step of kind 0: the links for F = TA(U G^dag); null otherwise
};

template <bool BWD, typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_loops(const __grid_constant__ StoutPlaqArgs<T> a)
{
    pdl_enter();
    const int x = blockIdx.x * kStoutBlock + threadIdx.x, V = a.g.V;
    if (x >= V) return;
    const int p = blockIdx.y;
    int m, n;
    plane_dirs(p, m, n);
    const int xm = up(a.g, x, m), xn = up(a.g, x, n);
    const M3T<T> pmn = mul<false, false>(link_at<T>(a.U, a.g, n, x), link_at<T>(a.U, a.g, m, xn));
    const M3T<T> pnm = mul<false, false>(link_at<T>(a.U, a.g, m, x), link_at<T>(a.U, a.g, n, xm));
    if (BWD) {
        ws_st(a.P, V, 2 * p, x, pmn);
        ws_st(a.P, V, 2 * p + 1, x, pnm);
    }
    ws_st9(a.K, V, p, x, anti_mul<false, true>(pmn, pnm));
    M3T<T> s = mul<true, false>(link_at<T>(a.U, a.g, n, x), pnm);  // Slo(m, n): of link (x+n, m)
    if (BWD) ws_st(a.Slo, V, 2 * p, x, s);
    ws_st9(a.Lo, V, 2 * p, x, anti_mul<false, true>(s, link_at<T>(a.U, a.g, m, xn)));
    s = mul<true, false>(link_at<T>(a.U, a.g, m, x), pmn);  // Slo(n, m): of link (x+m, n)
    if (BWD) ws_st(a.Slo, V, 2 * p + 1, x, s);
    ws_st9(a.Lo, V, 2 * p + 1, x, anti_mul<false, true>(s, link_at<T>(a.U, a.g, n, xm)));
}

// Q = -i TA(C U^dag) of link (x, mu) from its loops
template <typename T>
__device__ __forceinline__ plaq::H9<T> loops_q(const StoutPlaqArgs<T> &a, int mu, int x)
{
    H9<T> z;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        z.d[k] = T(0);
        z.o[k] = cx<T>{T(0), T(0)};
    }
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        axpy9(z, mu < nu ? T(1) : T(-1), ws_ld9(a.K, a.g.V, plane_of(mu, nu), x));
        axpy9(z, T(1), ws_ld9(a.Lo, a.g.V, slot_of(mu, nu), down(a.g, x, nu)));
    }
    return q_of(z, a.rho);
}

template <typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_apply(const __grid_constant__ StoutPlaqArgs<T> a)
{
    pdl_enter();
    const int mu = blockIdx.y, x = blockIdx.x * kStoutBlock + threadIdx.x;
    if (x >= a.g.V) return;
    const H9<T> q = loops_q(a, mu, x), q2 = square9(q);
    T c0, c1;
    char_coefs9(q, q2, c0, c1);
    const ExpCoefT<T> e = exp_sums<false>(c0, c1);
    const M3T<T> u = mul<false, false>(poly9(e.f, q, q2), link_at<T>(a.U, a.g, mu, x));
    st(a.out, a.g, mu, x, u);
}

// per link: E^dag G' into out, W and Y
template <typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_grad_exp(const __grid_constant__ StoutPlaqArgs<T> a)
{
    pdl_enter();
    const int mu = blockIdx.y, x = blockIdx.x * kStoutBlock + threadIdx.x, V = a.g.V;
    if (x >= V) return;
    M3T<T> gu;
    H9<T> w;
    const M3T<T> u = link_at<T>(a.U, a.g, mu, x);
    exp_gradient(loops_q(a, mu, x), u, link_at<T>(a.G, a.g, mu, x), a.rho, gu, w);
    st(a.out, a.g, mu, x, gu);
    ws_st9(a.W, V, mu, x, w);
    M3T<T> y = zero3<T>();
    anti_mul_acc(y, w, u);
    ws_st(a.Y, V, mu, x, y);
}

template <typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_bent(const __grid_constant__ StoutPlaqArgs<T> a)
{
    pdl_enter();
    const int x = blockIdx.x * kStoutBlock + threadIdx.x, V = a.g.V;
    if (x >= V) return;
    const int f = blockIdx.y;  // ordered pair (mu, nu)
    int mu, nu;
    plane_dirs(f >> 1, mu, nu);
    if (f & 1) { const int t = mu; mu = nu; nu = t; }
    H9<T> d = ws_ld9(a.W, V, nu, x);
    axpy9(d, T(-1), ws_ld9(a.W, V, mu, x));
    M3T<T> p = zero3<T>();
    anti_mul_acc(p, d, ws_ld<T>(a.P, V, f, x));
    mul_acc<false, false>(p, link_at<T>(a.U, a.g, nu, x), ws_ld<T>(a.Y, V, mu, up(a.g, x, nu)));
    ws_st(a.Pb, V, f, x, p);
}

template <typename T>
__global__ void __launch_bounds__(kStoutBlock) k_stout_gather(const __grid_constant__ StoutPlaqArgs<T> a)
{
    pdl_enter();
    const int mu = blockIdx.y, x = blockIdx.x * kStoutBlock + threadIdx.x, V = a.g.V;
    if (x >= V) return;
    const int xm = up(a.g, x, mu);
    M3T<T> G = link_at<T>(a.out, a.g, mu, x), S = zero3<T>();
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        const int f = slot_of(mu, nu), y = down(a.g, x, nu);
        axpy3(S, T(-1), ws_ld<T>(a.Slo, V, f, y));
        mul_acc<false, true>(G, ws_ld<T>(a.Pb, V, f, x), link_at<T>(a.U, a.g, nu, xm));
        mul_acc<false, true>(G, ws_ld<T>(a.P, V, f, x), ws_ld<T>(a.Y, V, nu, xm));
        mul_acc<true, false>(G, link_at<T>(a.U, a.g, nu, y), ws_ld<T>(a.Pb, V, f ^ 1, y));
    }
    anti_mul_acc(G, ws_ld9(a.W, V, mu, x), S);
    if (a.proj) G = expand_anti_traceless(anti_mul<false, true>(link_at<T>(a.proj, a.g, mu, x), G));
    st(a.out, a.g, mu, x, G);
}

stg_status check_common(const stg_lattice *lat, int nstep, double rho, const char *fn)
{
    const std::string f(fn);
    if (!lat) return set_error(STG_ERR_ARG, f + ": null lattice");
    if (lat->V > kMaxLinkSites) return set_error(STG_ERR_SHAPE, f + ": lattice of 2^31 sites");
    if (nstep < 1 || nstep > 16) return set_error(STG_ERR_ARG, f + ": nstep must be in 1..16");
    if (!(fabs(rho) <= 0.5)) return set_error(STG_ERR_ARG, f + ": |rho| must be <= 0.5");
    return STG_OK;
}

bool misaligned(const void *p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15) != 0; }

// Workspaces of the shared-plaquette steps: 1.3 kB (smearing) and 7.3 kB (chain rule) per site in
// FP64.  Beyond kStoutWorkspace, without room for them and while the stream captures, the per-link
// kernels above do the step.
constexpr size_t kStoutWorkspace = (size_t)8 << 30;

// Bump allocation of [count] fields of 9 V entries
template <typename E>
E *take(char *&p, int V, int count)
{
    E *r = reinterpret_cast<E *>(p);
    p += ((size_t)count * 9 * V * sizeof(E) + 255) & ~(size_t)255;
    return r;
}

// Whether the steps go by shared plaquettes: FP64 within the workspace.  FP32 stays with the per-link kernels,
// which are not bound by their products (32^4 chain rule: 2.8 ms against 5.1 ms shared).
template <typename T>
bool plaq_fits(size_t bytes)
{
    return sizeof(T) == 8 && bytes <= kStoutWorkspace;
}

// Smearing has one window of its own.  In FP64 every warp has a quarter SM's pipe to itself while a launch has
// no more warps than quarters; where the per-link kernel fits that once and the 6 planes of a site do not
// (3233 to 4864 sites on 152 SMs) it is faster: 8^4 130 us against 147 us, but 3072 sites 130 against 101, 5120
// 238 against 171.  The chain rule has none, its per-link kernels do nearly twice the products: 8^4 437 us
// against 329 us, 768 sites 426 against 250, 6400 812 against 472.
inline bool smear_by_links(long long V)
{
    const long long warps = (V + 31) / 32, quarters = 4LL * sm_count();
    return 6 * warps > quarters && 4 * warps <= quarters;
}

template <typename T>
bool smear_plaq(const stg_lattice *lat, int nstep, double rho, const void *links, void *levels, cudaStream_t st,
                cudaError_t &err)
{
    using C = typename C2<T>::type;
    const size_t bytes = (size_t)18 * 9 * lat->V * sizeof(T) + 4096;
    if (!plaq_fits<T>(bytes) || smear_by_links(lat->V)) return false;
    char *ws = nullptr, *w;
    if (link_workspace((void **)&ws, bytes, st) != cudaSuccess) return false;
    StoutPlaqArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = link_geo(lat->g);
    a.rho = (T)rho;
    w = ws;
    a.K = take<T>(w, a.g.V, 6);
    a.Lo = take<T>(w, a.g.V, 12);
    const size_t level = (size_t)4 * a.g.V * 9;
    const unsigned nb = (unsigned)((a.g.V + kStoutBlock - 1) / kStoutBlock);
    const bool ov = overlap(a.g.V, 10, 4, 26000);
    err = cudaSuccess;
    for (int k = 0; k < nstep && err == cudaSuccess; ++k) {
        a.U = k == 0 ? static_cast<const C *>(links) : static_cast<const C *>(levels) + (size_t)(k - 1) * level;
        a.out = static_cast<C *>(levels) + (size_t)k * level;
        err = launch_overlap(ov, k_stout_loops<false, T>, dim3(nb, 6), dim3(kStoutBlock), 0, st, a);
        if (err == cudaSuccess) err = launch_overlap(ov, k_stout_apply<T>, dim3(nb, 4), dim3(kStoutBlock), 0, st, a);
    }
    const cudaError_t f = cudaFreeAsync(ws, st);
    if (err == cudaSuccess) err = f;
    return true;
}

template <typename T>
bool force_plaq(const stg_lattice *lat, int nstep, double rho, const void *links, const void *levels, const void *grad,
                void *out_v, int kind, cudaStream_t st, cudaError_t &err)
{
    using C = typename C2<T>::type;
    const size_t level = (size_t)4 * lat->V * 9;
    const size_t bytes = (size_t)(22 * 9 + (36 + 4) * 18) * lat->V * sizeof(T) +
                         (nstep > 1 ? level * sizeof(C) : 0) + 4096;
    if (!plaq_fits<T>(bytes)) return false;
    char *ws = nullptr, *w;
    if (link_workspace((void **)&ws, bytes, st) != cudaSuccess) return false;
    StoutPlaqArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = link_geo(lat->g);
    a.rho = (T)rho;
    w = ws;
    a.K = take<T>(w, a.g.V, 6);
    a.Lo = take<T>(w, a.g.V, 12);
    a.W = take<T>(w, a.g.V, 4);
    a.P = take<C>(w, a.g.V, 12);
    a.Slo = take<C>(w, a.g.V, 12);
    a.Pb = take<C>(w, a.g.V, 12);
    a.Y = take<C>(w, a.g.V, 4);
    C *tmp = nstep > 1 ? take<C>(w, a.g.V, 4) : nullptr;
    C *out = static_cast<C *>(out_v);
    const unsigned nb = (unsigned)((a.g.V + kStoutBlock - 1) / kStoutBlock);
    const dim3 links4(nb, 4);
    const bool ov = overlap(a.g.V, 16, 4, 8192);
    a.G = static_cast<const C *>(grad);
    err = cudaSuccess;
    for (int k = nstep - 1; k >= 0 && err == cudaSuccess; --k) {
        // the last step (k = 0) lands in out; earlier ones alternate so that it does
        a.U = k == 0 ? static_cast<const C *>(links) : static_cast<const C *>(levels) + (size_t)(k - 1) * level;
        a.out = (k % 2 == 0) ? out : tmp;
        a.proj = k == 0 && kind == 0 ? static_cast<const C *>(links) : nullptr;
        err = launch_overlap(ov, k_stout_loops<true, T>, dim3(nb, 6), dim3(kStoutBlock), 0, st, a);
        if (err == cudaSuccess) err = launch_overlap(ov, k_stout_grad_exp<T>, links4, dim3(kStoutBlock), 0, st, a);
        if (err == cudaSuccess) err = launch_overlap(ov, k_stout_bent<T>, dim3(nb, 12), dim3(kStoutBlock), 0, st, a);
        if (err == cudaSuccess) err = launch_overlap(ov, k_stout_gather<T>, links4, dim3(kStoutBlock), 0, st, a);
        a.G = a.out;
    }
    const cudaError_t f = cudaFreeAsync(ws, st);
    if (err == cudaSuccess) err = f;
    return true;
}

// The per-link kernels, on canonical links.  The FP32 chain rule keeps its intermediate fields, and a
// copy of the links for the staple terms (k_links_to_ws), as workspace fields when there is room:
// 32^4 3.53 -> 2.97 ms, 16^4 266 -> 200 us (2.79 ms with the four directions of 32 sites in one block, which
// share links through L1; smearing 1.10 -> 1.01 ms).  Smearing and the first chain-rule kernel read the
// canonical links (a smearing step from the workspace form took 690 us against 550).
template <typename T>
cudaError_t smear_t(const LinkGeo &g, int nstep, double rho, const void *links, void *levels, cudaStream_t st)
{
    using C = typename C2<T>::type;
    StoutArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = g;
    a.rho = (T)rho;
    const size_t level = (size_t)4 * g.V * 9;  // complex numbers per level
    const dim3 grid((unsigned)((g.V + 31) / 32));  // 32 sites, one warp per direction
    const bool ov = sizeof(T) == 4 || overlap(g.V, 8, 4, 26000);
    for (int k = 0; k < nstep; ++k) {
        a.U = k == 0 ? static_cast<const C *>(links) : static_cast<const C *>(levels) + (size_t)(k - 1) * level;
        a.out = static_cast<C *>(levels) + (size_t)k * level;
        const cudaError_t e = launch_overlap(ov, k_stout_fwd<T>, grid, dim3(kStoutBlock), 0, st, a);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t force_t(const LinkGeo &g, int nstep, double rho, const void *links, const void *levels, const void *grad,
                    void *out_v, int kind, cudaStream_t st)
{
    using C = typename C2<T>::type;
    StoutArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = g;
    a.rho = (T)rho;
    const size_t level = (size_t)4 * g.V * 9;
    C *ws = nullptr;
    // without room, and while st captures, in the canonical form with two arrays of the default pool
    const bool soa = sizeof(T) == 4 && link_workspace((void **)&ws, 3 * level * sizeof(C), st) == cudaSuccess;
    cudaError_t e = soa ? cudaSuccess : cudaMallocAsync((void **)&ws, 2 * level * sizeof(C), st);
    if (e != cudaSuccess) return e;
    C *tmp = ws + level, *U = ws + 2 * level, *out = static_cast<C *>(out_v);
    a.Y = ws;
    const dim3 grid((unsigned)((g.V + 31) / 32)), block(kStoutBlock);  // 32 sites, one warp per direction
    const bool ov = sizeof(T) == 4 ? overlap(g.V, 8, 6, 16384) : overlap(g.V, 8, 4, 8192);
    a.G = static_cast<const C *>(grad);
    a.g_canon = 1;
    for (int k = nstep - 1; k >= 0 && e == cudaSuccess; --k) {
        a.U = k == 0 ? static_cast<const C *>(links) : static_cast<const C *>(levels) + (size_t)(k - 1) * level;
        a.proj = k == 0 && kind == 0;
        bool done = false;
        if constexpr (sizeof(T) == 4) {
            if (soa) {
                // each link's G, own terms and result share one place of tmp; the last result goes to out
                e = links_to_ws<T>(ov, a.U, U, g.V, st);
                a.Uws = U;
                a.acc = tmp;
                a.out = k == 0 ? out : tmp;
                a.out_canon = k == 0;
                if (e == cudaSuccess) e = launch_overlap(ov, k_stout_back_link<true, T>, grid, block, 0, st, a);
                if (e == cudaSuccess) e = launch_overlap(ov, k_stout_back_staples<true, T>, grid, block, 0, st, a);
                a.g_canon = 0;
                done = true;
            }
        }
        if (!done) {
            // the last step (k = 0) lands in out; earlier ones alternate so that it does
            a.acc = a.out = (k % 2 == 0) ? out : tmp;
            e = launch_overlap(ov, k_stout_back_link<false, T>, grid, block, 0, st, a);
            if (e == cudaSuccess) e = launch_overlap(ov, k_stout_back_staples<false, T>, grid, block, 0, st, a);
        }
        a.G = a.out;
    }
    const cudaError_t f = cudaFreeAsync(ws, st);
    return e != cudaSuccess ? e : f;
}

}  // namespace
}  // namespace stg

using namespace stg;

extern "C" stg_status stg_stout_smear(const stg_lattice *lat, stg_prec prec, int32_t nstep, double rho,
                                      const void *links_dev, void *levels_dev, void *stream)
{
    if (lat && stg::geom_is_slab(lat->g))
        return stg::set_error(STG_ERR_SHAPE, "stg_stout_smear: not available on a slab lattice (stg_dslash* only)");
    stg_status s = check_common(lat, nstep, rho, "stg_stout_smear");
    if (s != STG_OK) return s;
    if (prec != STG_F64 && prec != STG_F32) return set_error(STG_ERR_ARG, "stg_stout_smear: prec must be F64 or F32");
    if (misaligned(links_dev) || misaligned(levels_dev))
        return set_error(STG_ERR_ARG, "stg_stout_smear: buffers must be non-null and 16-byte aligned");
    const LinkGeo g = link_geo(lat->g);
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t err = cudaSuccess;
    if (prec == STG_F64 && smear_plaq<double>(lat, nstep, rho, links_dev, levels_dev, st, err)) {
        STG_CUDA_TRY(err);
        return STG_OK;
    }
    STG_CUDA_TRY(prec == STG_F64 ? smear_t<double>(g, nstep, rho, links_dev, levels_dev, st)
                                 : smear_t<float>(g, nstep, rho, links_dev, levels_dev, st));
    return STG_OK;
}

extern "C" stg_status stg_stout_force(const stg_lattice *lat, stg_prec prec, int32_t nstep, double rho,
                                      const void *links_dev, const void *levels_dev, const void *grad_dev,
                                      void *out_dev, int32_t kind, void *stream)
{
    if (lat && stg::geom_is_slab(lat->g))
        return stg::set_error(STG_ERR_SHAPE, "stg_stout_force: not available on a slab lattice (stg_dslash* only)");
    stg_status s = check_common(lat, nstep, rho, "stg_stout_force");
    if (s != STG_OK) return s;
    if (prec != STG_F64 && prec != STG_F32) return set_error(STG_ERR_ARG, "stg_stout_force: prec must be F64 or F32");
    if (misaligned(links_dev) || misaligned(grad_dev) || misaligned(out_dev) || (nstep > 1 && misaligned(levels_dev)))
        return set_error(STG_ERR_ARG, "stg_stout_force: buffers must be non-null and 16-byte aligned");
    if (kind != 0 && kind != 1) return set_error(STG_ERR_ARG, "stg_stout_force: kind must be 0 or 1");
    if (out_dev == grad_dev || out_dev == links_dev)
        return set_error(STG_ERR_ARG, "stg_stout_force: out must not alias the inputs");
    const LinkGeo g = link_geo(lat->g);
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t err = cudaSuccess;
    if (prec == STG_F64 &&
        force_plaq<double>(lat, nstep, rho, links_dev, levels_dev, grad_dev, out_dev, kind, st, err)) {
        STG_CUDA_TRY(err);
        return STG_OK;
    }
    STG_CUDA_TRY(prec == STG_F64 ? force_t<double>(g, nstep, rho, links_dev, levels_dev, grad_dev, out_dev, kind, st)
                                 : force_t<float>(g, nstep, rho, links_dev, levels_dev, grad_dev, out_dev, kind, st));
    return STG_OK;
}
