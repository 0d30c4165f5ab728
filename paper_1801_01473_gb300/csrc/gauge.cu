// gauge.cu -- the tree-level Symanzik gauge action S_g and its force (Sec. 2: S_g is built from
// the traces of 1x1 plaquettes and 1x2 rectangles of the unsmeared links; Sec. 3: the gauge term
// of the MD force needs the products of links along those loops, the "staples").
//
//   S_g = -(beta/3) sum_x sum_{mu != nu} [ c0 Re tr P_{mu nu}(x) + c1 Re tr R_{mu nu}(x) ]
//   c0 = 5/6, c1 = -1/12 (tree-level coefficients; ordered pairs: each plaquette twice, each
//   2x1 rectangle once), links periodic in all four directions.
//
// Force: for the link U_mu(x) every loop through it reads Re tr(U_mu(x) B) with B the rest of the
// loop, so G = dS/dRe U + i dS/dIm U = -(beta/3) sum c B^dag; B^dag is the "staple".  Per link:
// 2 plaquette staples (weight 2 c0) and 6 rectangle staples (weight c1) per direction nu != mu.
// Output kind 1: G; kind 0: F = TA(U G^dag) (dS/deps = tr(X F) along U -> exp(eps X) U).
//
// Canonical complex128 [4][V][3][3]; FP64 forces share their staples between links, FP32 ones are
// one thread per link over its loops (84 complex 3x3 products).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "dslash.cuh"
#include "plaq.cuh"
#include "stg_common.h"
#include "su3.cuh"

namespace stg {
namespace {
using namespace su3;

constexpr double kC0 = 5.0 / 6.0, kC1 = -1.0 / 12.0;
constexpr int kGaugeBlock = 128;

template <typename T>
struct GaugeArgs {
    using C = typename C2<T>::type;
    LinkGeo g;
    double beta;
    const C *U;
    C *out;
    int kind;
    double *partial;  // action: [2][nblocks] (plaquette sums, rectangle sums)
    double *out3;     // action: S_g, plaquette sum, rectangle sum
    int nblocks;
};

template <typename T>
__device__ __forceinline__ M3T<T> lk(const typename C2<T>::type *__restrict__ U, const LinkGeo &g, int d,
                                     int site)
{
    M3T<T> m;
    ld(U, g, d, site, m);
    return m;
}

// Re tr(a b)
__device__ __forceinline__ double retr_mul(const M3 &a, const M3 &b)
{
    double s = 0.0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) s += a.m[r][k].re * b.m[k][r].re - a.m[r][k].im * b.m[k][r].im;
    return s;
}

// Re tr(a b^dag)
__device__ __forceinline__ double retr_mul_dag(const M3 &a, const M3 &b)
{
    double s = 0.0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) s = fma(a.m[r][k].im, b.m[r][k].im, fma(a.m[r][k].re, b.m[r][k].re, s));
    return s;
}

// G = wr [sum of rectangle staples + kPlaq * sum of plaquette staples], kPlaq = 2 c0 / c1.  Each side
// (upper, lower) of a plane is one plaquette staple U_nu U_mu U_nu^dag (lower: U_nu^dag U_mu U_nu) and
// its three forms with one factor replaced by that link's outer staple: 11 products a side (each summed
// before it is added to the larger total, which keeps the rounding of the loop-by-loop form), 66 per
// link (84 when every loop is multiplied out).  Bound by latency at two blocks of 250 registers per SM;
// three blocks of 168 ran 3 % slower at 32^4, four spill.  FP32, 32^4: 2.79 -> 1.86 ms with 32-bit site
// arithmetic (neighbours by multiplication instead of 64-bit division); 1.71 ms with the four directions
// of 32 sites in one block, which share the links of their staples through L1 (one direction per
// grid row re-read them from L2).  16^4: 182 -> 118 us.
template <typename T>
__global__ void __launch_bounds__(kGaugeBlock, 2) k_gauge_force(const __grid_constant__ GaugeArgs<T> a)
{
    const int mu = threadIdx.x >> 5;  // warp-uniform
    const int x = blockIdx.x * 32 + (threadIdx.x & 31);
    if (x >= a.g.V) return;
    const LinkGeo &g = a.g;
    const typename C2<T>::type *__restrict__ Ub = a.U;
    const T wr = T(-a.beta / 3.0 * kC1), kPlaq = T(2.0 * kC0 / kC1);
    M3T<T> G = zero3<T>();
    const int xpm = up(g, x, mu), xmm = down(g, x, mu), xp2m = up(g, xpm, mu);
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        M3T<T> t, s, X;
        {
            const int xpn = up(g, x, nu), xpm_pn = up(g, xpm, nu);
            // U_nu(x) U_mu(x+nu), with the outer staple of the last factor U_nu(x+mu)^dag
            t = mul<false, false>(lk<T>(Ub, g, nu, x), lk<T>(Ub, g, mu, xpn));
            s = mul<false, true>(lk<T>(Ub, g, mu, xpm_pn), lk<T>(Ub, g, nu, xp2m));
            s = mul<false, true>(s, lk<T>(Ub, g, mu, xpm));
            plaq::axpy3(G, T(1), mul<false, false>(t, s));
            // outer staple of the middle factor U_mu(x+nu)
            s = mul<false, false>(lk<T>(Ub, g, nu, xpn), lk<T>(Ub, g, mu, up(g, xpn, nu)));
            s = mul<false, true>(s, lk<T>(Ub, g, nu, xpm_pn));
            X = mul<false, false>(lk<T>(Ub, g, nu, x), s);
            // outer staple of the first factor U_nu(x)
            s = mul<true, false>(lk<T>(Ub, g, mu, xmm), lk<T>(Ub, g, nu, xmm));
            s = mul<false, false>(s, lk<T>(Ub, g, mu, up(g, xmm, nu)));
            mul_acc<false, false>(X, s, lk<T>(Ub, g, mu, xpn));
            plaq::axpy3(X, kPlaq, t);
            plaq::axpy3(G, T(1), mul<false, true>(X, lk<T>(Ub, g, nu, xpm)));
        }
        {
            const int xmn = down(g, x, nu), xpm_mn = down(g, xpm, nu), xm2n = down(g, xmn, nu), xmm_mn = down(g, xmm, nu);
            // U_nu(x-nu)^dag U_mu(x-nu), with the outer staple of the last factor U_nu(x+mu-nu)
            t = mul<true, false>(lk<T>(Ub, g, nu, xmn), lk<T>(Ub, g, mu, xmn));
            s = mul<false, false>(lk<T>(Ub, g, mu, xpm_mn), lk<T>(Ub, g, nu, down(g, xp2m, nu)));
            s = mul<false, true>(s, lk<T>(Ub, g, mu, xpm));
            plaq::axpy3(G, T(1), mul<false, false>(t, s));
            // outer staple of the middle factor U_mu(x-nu)
            s = mul<true, false>(lk<T>(Ub, g, nu, xm2n), lk<T>(Ub, g, mu, xm2n));
            s = mul<false, false>(s, lk<T>(Ub, g, nu, down(g, xpm_mn, nu)));
            X = mul<true, false>(lk<T>(Ub, g, nu, xmn), s);
            // outer staple of the first factor U_nu(x-nu)^dag
            s = mul<true, true>(lk<T>(Ub, g, mu, xmm), lk<T>(Ub, g, nu, xmm_mn));
            s = mul<false, false>(s, lk<T>(Ub, g, mu, xmm_mn));
            mul_acc<false, false>(X, s, lk<T>(Ub, g, mu, xmn));
            plaq::axpy3(X, kPlaq, t);
            plaq::axpy3(G, T(1), mul<false, false>(X, lk<T>(Ub, g, nu, xpm_mn)));
        }
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) G.m[r][c] = cx<T>{wr * G.m[r][c].re, wr * G.m[r][c].im};
    if (a.kind == 0) G = plaq::expand_anti_traceless(plaq::anti_mul<false, true>(lk<T>(Ub, g, mu, x), G));
    st(a.out, g, mu, x, G);
}

// ------------------------------------------------------------------ force by shared staples
// The 2x1 rectangle across link (y, nu) is tr[Sup(nu, mu)(y) Slo(nu, mu)(y-mu)^dag], the product of
// the link's upper and lower staples (plaq.cuh).  So the rectangle part of the force is the plaquette
// part with one link of the plaquette replaced by its staple on the outer side:
//   P'(mu, nu)(x) = Slo(nu, mu)(x-mu) U_mu(x+nu) + U_nu(x) Sup(mu, nu)(x+nu)
//   G_mu(x) = sum_nu  wp Sup(mu, nu)(x) + wr [ P'(mu, nu)(x) U_nu(x+mu)^dag + P(mu, nu)(x) Sup(nu, mu)(x+mu)^dag ]
//                   + wp Slo(mu, nu)(y) + wr [ U_nu(y)^dag P'(nu, mu)(y) + Slo(nu, mu)(y-mu)^dag P(nu, mu)(y) ]
// with y = x - nu.  Three products per ordered pair for P, Sup, Slo (k_gauge_staples), two for P'
// (k_gauge_bent), four per link and nu for G (k_gauge_gather): 27 products per link where the loops
// one by one take 84 (k_gauge_force), for 4 matrices of workspace per pair and site.
// Bound by the FP64 pipe: 18x22x14x26 8.73 -> 3.02 ms (2970 multiply-adds per link at 0.57e12/s),
// 24^4 20.0 -> 6.93 ms, 4^4 317 -> 77 us.  One warp per block: the pipe is per quarter SM and one warp
// keeps it busy, so small lattices spread best in single warps (6^4, overlapping launches: 98 us against 123 us
// with four; launched plainly, as it is now, 86 us).
constexpr int kPlaqBlock = 32;

template <typename T>
struct GaugePlaqArgs {
    using C = typename C2<T>::type;
    LinkGeo g;
    const C *U;
    C *P, *Sup, *Slo, *Pb;  // one field per ordered pair of the planes [p0, p1)
    C *out;
    T wp, wr;
    int p0, p1;  // planes of this pass
    int first, last, kind;
};

template <typename T>
__global__ void __launch_bounds__(kPlaqBlock) k_gauge_staples(const __grid_constant__ GaugePlaqArgs<T> a)
{
    using namespace plaq;
    pdl_enter();
    const int x = blockIdx.x * kPlaqBlock + threadIdx.x;
    if (x >= a.g.V) return;
    int mu, nu;
    plane_dirs(a.p0 + (blockIdx.y >> 1), mu, nu);
    if (blockIdx.y & 1) { const int t = mu; mu = nu; nu = t; }
    const int f = blockIdx.y;
    const M3T<T> p = mul<false, false>(link_at<T>(a.U, a.g, nu, x), link_at<T>(a.U, a.g, mu, up(a.g, x, nu)));
    ws_st(a.P, a.g.V, f, x, p);
    ws_st(a.Sup, a.g.V, f, x, mul<false, true>(p, link_at<T>(a.U, a.g, nu, up(a.g, x, mu))));
    ws_st(a.Slo, a.g.V, f ^ 1, x, mul<true, false>(link_at<T>(a.U, a.g, mu, x), p));
}

template <typename T>
__global__ void __launch_bounds__(kPlaqBlock) k_gauge_bent(const __grid_constant__ GaugePlaqArgs<T> a)
{
    using namespace plaq;
    pdl_enter();
    const int x = blockIdx.x * kPlaqBlock + threadIdx.x;
    if (x >= a.g.V) return;
    int mu, nu;
    plane_dirs(a.p0 + (blockIdx.y >> 1), mu, nu);
    if (blockIdx.y & 1) { const int t = mu; mu = nu; nu = t; }
    const int f = blockIdx.y, xn = up(a.g, x, nu);
    M3T<T> p = mul<false, false>(ws_ld<T>(a.Slo, a.g.V, f ^ 1, down(a.g, x, mu)), link_at<T>(a.U, a.g, mu, xn));
    mul_acc<false, false>(p, link_at<T>(a.U, a.g, nu, x), ws_ld<T>(a.Sup, a.g.V, f, xn));
    ws_st(a.Pb, a.g.V, f, x, p);
}

template <typename T>
__global__ void __launch_bounds__(kPlaqBlock) k_gauge_gather(const __grid_constant__ GaugePlaqArgs<T> a)
{
    using namespace plaq;
    pdl_enter();
    const int mu = blockIdx.y, x = blockIdx.x * kPlaqBlock + threadIdx.x;
    if (x >= a.g.V) return;
    const int V = a.g.V, xm = up(a.g, x, mu);
    M3T<T> G = zero3<T>(), R = zero3<T>();
    if (!a.first) G = link_at<T>(a.out, a.g, mu, x);
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == mu) continue;
        const int p = plane_of(mu, nu);
        if (p < a.p0 || p >= a.p1) continue;
        const int f = slot_of(mu, nu) - 2 * a.p0;  // pair (mu, nu); (nu, mu) is f ^ 1
        const int y = down(a.g, x, nu), ym = down(a.g, y, mu);
        axpy3(G, a.wp, ws_ld<T>(a.Sup, V, f, x));
        axpy3(G, a.wp, ws_ld<T>(a.Slo, V, f, y));
        mul_acc<false, true>(R, ws_ld<T>(a.Pb, V, f, x), link_at<T>(a.U, a.g, nu, xm));
        mul_acc<false, true>(R, ws_ld<T>(a.P, V, f, x), ws_ld<T>(a.Sup, V, f ^ 1, xm));
        mul_acc<true, false>(R, link_at<T>(a.U, a.g, nu, y), ws_ld<T>(a.Pb, V, f ^ 1, y));
        mul_acc<true, false>(R, ws_ld<T>(a.Slo, V, f ^ 1, ym), ws_ld<T>(a.P, V, f ^ 1, y));
    }
    axpy3(G, a.wr, R);
    if (a.last && a.kind == 0) G = expand_anti_traceless(anti_mul<false, true>(link_at<T>(a.U, a.g, mu, x), G));
    st(a.out, a.g, mu, x, G);
}

// Action from the same staples: the plaquette of a plane is Re tr[P(m, n) P(n, m)^dag], the rectangle
// across link (x, mu) in direction nu Re tr[Sup(mu, nu)(x) Slo(mu, nu)(x-nu)^dag], 18 multiply-adds each
// where k_gauge_action takes 10 products a plane.  One thread per site over the planes of the pass.
__global__ void __launch_bounds__(kGaugeBlock) k_gauge_traces(const __grid_constant__ GaugePlaqArgs<double> a,
                                                              double *partial)
{
    using namespace plaq;
    pdl_enter();
    __shared__ double sh[33];
    const int x = blockIdx.x * kGaugeBlock + threadIdx.x, V = a.g.V;
    double ps = 0.0, rs = 0.0;
    if (x < V) {
#pragma unroll 1
        for (int p = a.p0; p < a.p1; ++p) {
            int m, n;
            plane_dirs(p, m, n);
            const int f = 2 * (p - a.p0);
            ps += retr_mul_dag(ws_ld<double>(a.P, V, f, x), ws_ld<double>(a.P, V, f + 1, x));
            rs += retr_mul_dag(ws_ld<double>(a.Sup, V, f, x), ws_ld<double>(a.Slo, V, f, down(a.g, x, n)));
            rs += retr_mul_dag(ws_ld<double>(a.Sup, V, f + 1, x), ws_ld<double>(a.Slo, V, f + 1, down(a.g, x, m)));
        }
    }
    ps = block_sum(ps, sh);
    __syncthreads();
    rs = block_sum(rs, sh);
    if (threadIdx.x == 0) {
        double *q = partial + blockIdx.x;
        q[0] = a.first ? ps : q[0] + ps;
        q[gridDim.x] = a.first ? rs : q[gridDim.x] + rs;
    }
}

__global__ void __launch_bounds__(kGaugeBlock, 1) k_gauge_action(const __grid_constant__ GaugeArgs<double> a)
{
    __shared__ double sh[33];
    const int x = blockIdx.x * kGaugeBlock + threadIdx.x;
    const LinkGeo g = a.g;
    const double2 *__restrict__ Ub = a.U;
    double ps = 0.0, rs = 0.0;
    if (x < g.V) {
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu) {
            const int xpm = up(g, x, mu);
#pragma unroll 1
            for (int nu = mu + 1; nu < 4; ++nu) {
                const int xpn = up(g, x, nu);
                // P = U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
                M3 t = mul<false, false>(lk<double>(Ub, g, mu, x), lk<double>(Ub, g, nu, xpm));
                M3 w = mul<true, true>(lk<double>(Ub, g, mu, xpn), lk<double>(Ub, g, nu, x));
                ps += retr_mul(t, w);
                // R_{mu nu} = U_mu(x) U_mu(x+mu) U_nu(x+2mu) U_mu(x+mu+nu)^dag U_mu(x+nu)^dag U_nu(x)^dag
                t = mul<false, false>(lk<double>(Ub, g, mu, x), lk<double>(Ub, g, mu, xpm));
                t = mul<false, false>(t, lk<double>(Ub, g, nu, up(g, xpm, mu)));
                w = mul<true, true>(lk<double>(Ub, g, mu, up(g, xpm, nu)), lk<double>(Ub, g, mu, xpn));
                w = mul<false, true>(w, lk<double>(Ub, g, nu, x));
                rs += retr_mul(t, w);
                // R_{nu mu} = U_nu(x) U_nu(x+nu) U_mu(x+2nu) U_nu(x+nu+mu)^dag U_nu(x+mu)^dag U_mu(x)^dag
                t = mul<false, false>(lk<double>(Ub, g, nu, x), lk<double>(Ub, g, nu, xpn));
                t = mul<false, false>(t, lk<double>(Ub, g, mu, up(g, xpn, nu)));
                w = mul<true, true>(lk<double>(Ub, g, nu, up(g, xpn, mu)), lk<double>(Ub, g, nu, xpm));
                w = mul<false, true>(w, lk<double>(Ub, g, mu, x));
                rs += retr_mul(t, w);
            }
        }
    }
    ps = block_sum(ps, sh);
    __syncthreads();
    rs = block_sum(rs, sh);
    if (threadIdx.x == 0) {
        a.partial[blockIdx.x] = ps;
        a.partial[a.nblocks + blockIdx.x] = rs;
    }
}

// fixed-order sum of the block partials by one block; writes S_g, plaquette sum, rectangle sum
__global__ void __launch_bounds__(256) k_gauge_action_finish(const __grid_constant__ GaugeArgs<double> a)
{
    __shared__ double sh[33];
    double ps = 0.0, rs = 0.0;
    for (int k = threadIdx.x; k < a.nblocks; k += blockDim.x) {
        ps += a.partial[k];
        rs += a.partial[a.nblocks + k];
    }
    ps = block_sum(ps, sh);
    __syncthreads();
    rs = block_sum(rs, sh);
    if (threadIdx.x == 0) {
        // sum over ordered pairs: each plaquette twice (ps counts it once), each rectangle once
        a.out3[0] = -a.beta / 3.0 * (2.0 * kC0 * ps + kC1 * rs);
        a.out3[1] = ps;
        a.out3[2] = rs;
    }
}

bool misaligned(const void *p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15) != 0; }

}  // namespace
}  // namespace stg

using namespace stg;

// Workspace of the shared-staple force and action: as many planes per pass as fit kGaugeWorkspace (all 6 up to
// 24^4 in the force), at least one (1152 bytes per site for the force, 864 for the action: 6.1 GB at 48^4).
constexpr size_t kGaugeWorkspace = (size_t)4 << 30;

// The planes per pass and the workspace of `fields` matrices per plane and site; false when there is
// no room for one plane, and while st captures: the kernels that need none then do the work.
template <typename C>
static bool plaq_workspace(long long V, int fields, cudaStream_t st, int &np, C *&ws)
{
    const size_t per_plane = (size_t)fields * 9 * V * sizeof(C);
    np = (int)std::min<size_t>(6, std::max<size_t>(1, kGaugeWorkspace / per_plane));
    cudaError_t e = link_workspace((void **)&ws, np * per_plane, st);
    if (e == cudaErrorMemoryAllocation && np > 1) {
        np = 1;
        e = link_workspace((void **)&ws, per_plane, st);
    }
    return e == cudaSuccess;
}

template <typename T>
static bool gauge_force_plaq(const stg_lattice *lat, double beta, const void *links, void *out, int kind,
                             cudaStream_t st, cudaError_t &err)
{
    using C = typename C2<T>::type;
    GaugePlaqArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = link_geo(lat->g);
    a.U = static_cast<const C *>(links);
    a.out = static_cast<C *>(out);
    a.wp = T(-beta / 3.0 * 2.0 * kC0);
    a.wr = T(-beta / 3.0 * kC1);
    a.kind = kind;
    int np = 0;
    C *ws = nullptr;
    if (!plaq_workspace(lat->V, 8, st, np, ws)) return false;
    err = cudaSuccess;
    const size_t field = (size_t)9 * a.g.V;
    a.P = ws;
    a.Sup = ws + 2 * np * field;
    a.Slo = ws + 4 * np * field;
    a.Pb = ws + 6 * np * field;
    const unsigned nb = (unsigned)((a.g.V + kPlaqBlock - 1) / kPlaqBlock);
    const bool ov = plaq::overlap(a.g.V, 24, 4, 8192);
    for (int p = 0; p < 6 && err == cudaSuccess; p += np) {
        a.p0 = p;
        a.p1 = std::min(6, p + np);
        a.first = p == 0;
        a.last = a.p1 == 6;
        const dim3 pairs(nb, 2 * (a.p1 - a.p0));
        err = launch_overlap(ov, k_gauge_staples<T>, pairs, dim3(kPlaqBlock), 0, st, a);
        if (err == cudaSuccess) err = launch_overlap(ov, k_gauge_bent<T>, pairs, dim3(kPlaqBlock), 0, st, a);
        if (err == cudaSuccess) err = launch_overlap(ov, k_gauge_gather<T>, dim3(nb, 4), dim3(kPlaqBlock), 0, st, a);
    }
    const cudaError_t f = cudaFreeAsync(ws, st);
    if (err == cudaSuccess) err = f;
    return true;
}

template <typename T>
static cudaError_t gauge_force_t(const stg_lattice *lat, double beta, const void *links, void *out, int kind,
                                 cudaStream_t st)
{
    cudaError_t err = cudaSuccess;
    GaugeArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = link_geo(lat->g);
    a.beta = beta;
    a.U = static_cast<const typename C2<T>::type *>(links);
    a.out = static_cast<typename C2<T>::type *>(out);
    a.kind = kind;
    // FP64: the shared staples wherever they fit (figures at the kernels).
    // FP32: the loops one by one, which need no workspace traffic (32^4: 1.71 ms against 2.77 ms shared)
    if constexpr (sizeof(T) == 8) {
        if (gauge_force_plaq<T>(lat, beta, links, out, kind, st, err)) return err;
    }
    const unsigned grid = (unsigned)((a.g.V + 31) / 32);  // 32 sites, one warp per direction
    k_gauge_force<T><<<grid, kGaugeBlock, 0, st>>>(a);
    return cudaGetLastError();
}

extern "C" stg_status stg_gauge_force(const stg_lattice *lat, stg_prec prec, double beta, const void *links_dev,
                                      void *out_dev, int32_t kind, void *stream)
{
    if (lat && stg::geom_is_slab(lat->g))
        return stg::set_error(STG_ERR_SHAPE, "stg_gauge_force: not available on a slab lattice (stg_dslash* only)");
    if (!lat) return set_error(STG_ERR_ARG, "stg_gauge_force: null lattice");
    if (lat->V > kMaxLinkSites) return set_error(STG_ERR_SHAPE, "stg_gauge_force: lattice of 2^31 sites");
    if (prec != STG_F64 && prec != STG_F32) return set_error(STG_ERR_ARG, "stg_gauge_force: prec must be F64 or F32");
    if (misaligned(links_dev) || misaligned(out_dev))
        return set_error(STG_ERR_ARG, "stg_gauge_force: buffers must be non-null and 16-byte aligned");
    if (out_dev == links_dev) return set_error(STG_ERR_ARG, "stg_gauge_force: out must not alias the links");
    if (kind != 0 && kind != 1) return set_error(STG_ERR_ARG, "stg_gauge_force: kind must be 0 or 1");
    if (!std::isfinite(beta)) return set_error(STG_ERR_ARG, "stg_gauge_force: beta must be finite");
    cudaStream_t st = (cudaStream_t)stream;
    STG_CUDA_TRY(prec == STG_F64 ? gauge_force_t<double>(lat, beta, links_dev, out_dev, kind, st)
                                 : gauge_force_t<float>(lat, beta, links_dev, out_dev, kind, st));
    return STG_OK;
}

extern "C" stg_status stg_gauge_action(const stg_lattice *lat, double beta, const void *links_c128_dev, double *out3_dev,
                                       void *stream)
{
    if (lat && stg::geom_is_slab(lat->g))
        return stg::set_error(STG_ERR_SHAPE, "stg_gauge_action: not available on a slab lattice (stg_dslash* only)");
    if (!lat) return set_error(STG_ERR_ARG, "stg_gauge_action: null lattice");
    if (lat->V > kMaxLinkSites) return set_error(STG_ERR_SHAPE, "stg_gauge_action: lattice of 2^31 sites");
    if (misaligned(links_c128_dev)) return set_error(STG_ERR_ARG, "stg_gauge_action: links must be non-null and 16-byte aligned");
    if (!out3_dev || (reinterpret_cast<uintptr_t>(out3_dev) & 7))
        return set_error(STG_ERR_ARG, "stg_gauge_action: out3 must be non-null and 8-byte aligned");
    if (!std::isfinite(beta)) return set_error(STG_ERR_ARG, "stg_gauge_action: beta must be finite");
    cudaStream_t st = (cudaStream_t)stream;
    GaugeArgs<double> a;
    memset(&a, 0, sizeof(a));
    a.g = link_geo(lat->g);
    a.beta = beta;
    a.U = static_cast<const double2 *>(links_c128_dev);
    a.out3 = out3_dev;
    a.nblocks = (int)((a.g.V + kGaugeBlock - 1) / kGaugeBlock);
    STG_CUDA_TRY(cudaMallocAsync((void **)&a.partial, 2 * sizeof(double) * a.nblocks, st));
    GaugePlaqArgs<double> q;
    memset(&q, 0, sizeof(q));
    int np = 0;
    double2 *ws = nullptr;
    if (plaq_workspace(lat->V, 6, st, np, ws)) {
        const size_t field = (size_t)9 * a.g.V;
        q.g = a.g;
        q.U = a.U;
        q.P = ws;
        q.Sup = ws + 2 * np * field;
        q.Slo = ws + 4 * np * field;
        cudaError_t e = cudaSuccess;
        for (int p = 0; p < 6 && e == cudaSuccess; p += np) {
            q.p0 = p;
            q.p1 = std::min(6, p + np);
            q.first = p == 0;
            const dim3 pairs((unsigned)((a.g.V + kPlaqBlock - 1) / kPlaqBlock), 2 * (q.p1 - q.p0));
            e = launch_pdl(k_gauge_staples<double>, pairs, dim3(kPlaqBlock), st, q);
            if (e == cudaSuccess) e = launch_pdl(k_gauge_traces, dim3(a.nblocks), dim3(kGaugeBlock), st, q, a.partial);
        }
        cudaFreeAsync(ws, st);
        if (e != cudaSuccess) {
            cudaFreeAsync(a.partial, st);
            STG_CUDA_TRY(e);
        }
    } else {
        k_gauge_action<<<a.nblocks, kGaugeBlock, 0, st>>>(a);
    }
    k_gauge_action_finish<<<1, 256, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(a.partial, st);
    STG_CUDA_TRY(e);
    return STG_OK;
}
