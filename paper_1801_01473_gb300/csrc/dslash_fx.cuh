// dslash_fx.cuh -- the hopping term on FP64 18-real links with its products on the integer pipes.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM, so the 288 products of an output site bind
// the FP64 operator at a third of the memory bandwidth.  The integer pipes multiply 32 x 32 -> 64 bits
// with a 64-bit accumulator at ~30 per clock and SM (measured), so three of those per product are
// faster.  Links (|U| < 2, unit 2^-55, laid out once per gauge) and the neighbour vectors of a site
// (unit 2^-55 of the power of two at or above the largest of them) are 57-bit signed fixed-point
// numbers in two limbs, value = l1 2^28 + l0 with |l0| <= 2^27, |l1| <= 2^28, and
//   sum u v = 2^56 sum u1 v1 + 2^28 sum (u1 v0 + u0 v1)      (u0 v0 is dropped)
// with both sums exact in 64 bits (48 terms of at most 2^56, 96 of at most 2^55).  Error of an
// output, with B the power of two above the largest component of the 8 neighbours: ~2^-55 B rms from
// the dropped term, the limbs' rounding and the final rounding together, against ~2^-53 B for the
// FP64 chain of 48 rounded multiply-adds (whole operator on the exp(0.3 i H) links: 1.46e-16 against
// 1.62e-16 of the 64-bit reference).  Links of 2 and above, infinities, NaNs, subnormal numbers and
// vectors near the ends of the exponent range go through the FP64 loop, thread by thread.
// D at 32^4 312 -> 152 us (of 100 us at the copy bandwidth), 24^4 108 -> 57 us, 16^4 46 -> 15 us, 8^4 15 ->
// 10 us.  What bounds it now: the integer pipes (864 products and ~1400 other operations a site; at
// 24^4 the multiply pipe is 57 % and the ALU 41 % busy) and, with one thread per site, loads in flight
// at 16 to 20 warps per SM.
#pragma once

#include "dslash.cuh"

namespace stg {

struct FxNum {
    int l1, l0;
};

__device__ __forceinline__ FxNum fx_split(long long w)
{
    w += 1 << 27;  // rounds the high limb: the low one is balanced around zero
    FxNum r;
    r.l1 = (int)(w >> 28);
    r.l0 = (int)((unsigned)w & 0xfffffffu) - (1 << 27);
    return r;
}

// d in units of 2^(E - 1078), truncated, for |d| < 2^(E - 1022) (E a biased exponent)
__device__ __forceinline__ FxNum fx_limbs(double d, int E)
{
    const int hi = __double2hiint(d);
    const unsigned lo = (unsigned)__double2loint(d);
    // (E << 20 | 0xfffff) - |hi| has E - e in its top bits (e the exponent of d)
    const int k = ((E << 20 | 0xfffff) - (hi & 0x7fffffff)) >> 20;
    const unsigned mh = (__funnelshift_l(lo, (unsigned)hi, 10) & 0x3fffffffu) | 0x40000000u;  // significand from bit 62
    const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 10);
    const long long v = (long long)(m >> min(k + 7, 63));
    const long long sg = (long long)(hi >> 31);
    return fx_split((v ^ sg) - sg);
}

__device__ __forceinline__ void fx_mac(long long &hh, long long &mid, const FxNum &a, const FxNum &b)
{
    hh += (long long)a.l1 * b.l1;
    mid += (long long)a.l1 * b.l0;
    mid += (long long)a.l0 * b.l1;
}

__device__ __forceinline__ FxNum fx_neg(const FxNum &a) { return FxNum{-a.l1, -a.l0}; }

// x 2^-d rounded, 0 <= d
__device__ __forceinline__ long long fx_shift(long long x, int d)
{
    d = min(d, 62);
    return (x + ((1ll << d) >> 1)) >> d;
}

// |d| < 2 (false for NaN), and d 2^55 rounded, both on the integer pipes: in FP64 the copy of a gauge
// was bound by the multiplications and conversions
__device__ __forceinline__ bool fx_below_two(double d) { return (__double2hiint(d) & 0x7fffffff) < 0x40000000; }
__device__ __forceinline__ long long fx_round55(double d)
{
    const int hi = __double2hiint(d);
    const int e = (hi & 0x7fffffff) >> 20;  // d = significand 2^(e - 1075)
    const long long m = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(d);
    const int s = 1020 - e;  // significand 2^(e - 1075 + 55)
    const long long v = s <= 0 ? m << -s : fx_shift(m, s);  // s >= -3: below 2^56
    return hi < 0 ? -v : v;
}

// Fixed-point links: per (mu, parity) block 9 chunks over Vh of (re.l1, re.l0, im.l1, im.l0)
struct LinkFX {
    static constexpr int kBytes = 144;
    __device__ __forceinline__ static void load(const void *blk, int Vh, int h, FxNum u[3][3][2])
    {
        const int4 *p = static_cast<const int4 *>(blk);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int4 q = __ldg(p + (size_t)k * Vh + h);
            u[k / 3][k % 3][0] = FxNum{q.x, q.y};
            u[k / 3][k % 3][1] = FxNum{q.z, q.w};
        }
    }
    // false when an entry has no fixed-point form
    __device__ __forceinline__ static bool pack(void *blk, int Vh, int h, const double2 *m)
    {
        int4 *p = static_cast<int4 *>(blk);
        bool ok = true;
        for (int k = 0; k < 9; ++k) {
            ok &= fx_below_two(m[k].x) && fx_below_two(m[k].y);
            const FxNum re = fx_split(ok ? fx_round55(m[k].x) : 0), im = fx_split(ok ? fx_round55(m[k].y) : 0);
            p[(size_t)k * Vh + h] = make_int4(re.l1, re.l0, im.l1, im.l0);
        }
        return ok;
    }
};

// acc += sign U v (or U^dag v) in FP64
template <bool BACK>
__device__ __forceinline__ void dp_hop(cx<double> acc[3], const cx<double> U[3][3], const cx<double> v[3], float sign)
{
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        cx<double> w = cx<double>{0.0, 0.0};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (BACK)
                cmac_conj(w, U[c][r], v[c]);
            else
                cmac(w, U[r][c], v[c]);
        }
        acc[r].re = fma((double)sign, w.re, acc[r].re);
        acc[r].im = fma((double)sign, w.im, acc[r].im);
    }
}

// One thread per output site.  Blocks of 64 threads keep 128 registers, larger ones 96 with a few
// spills: 24^4 58.7 -> 57.0 us with the higher occupancy.
template <int MODE, int BS>
__global__ void __launch_bounds__(BS, (BS == 64 ? 512 : 640) / BS) k_dslash_fx(const __grid_constant__ DArgs a)
{
    pdl_enter();
    const int bx = block_along_sites();
    const DGroup &G = a.grp[blockIdx.x];
    const int Vh = G.g.Vh;
    if (bx * BS >= G.g.h_end - G.g.h_begin) return;  // block-uniform
    if (G.nrhs < 1 || (G.skip[0] != nullptr && *G.skip[0] != 0)) return;  // block-uniform

    const int h = G.g.h_begin + bx * BS + threadIdx.x;
    const bool live = h < G.g.h_end;
    const int op = a.out_par;
    cx<double> acc[1][3];

    if (live) {
        const Site s = site_of(G.g, op, h);
        long long hh[3][2], mid[3][2];
        int E = 0;  // exponent of the unit's power of two; 0 while all neighbours were zero
        bool ok = *G.fx_bad == 0;
#pragma unroll
        for (int r = 0; r < 3; ++r) hh[r][0] = hh[r][1] = mid[r][0] = mid[r][1] = 0;
        // one direction per turn: all four unrolled are ~64 KB of instructions and ran slower
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu) {
            const Hop hp = hop_of(G.g, s, mu);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool back = k == 1;
                const int vi = back ? hp.hb : hp.hf;
                const bool flip = back ? hp.sb > 0.f : hp.sf < 0.f;  // the backward hop enters with -u
                FxNum u[3][3][2];
                LinkFX::load(link_block<LinkFX>(G.fx_links, Vh, mu, back ? 1 - op : op), Vh, back ? hp.hb : h, u);
                cx<double> v[3];
                Field<double>::load(G.in[0], Vh, vi, v);
                int e = 0;
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    e = max(e, max(__double2hiint(v[c].re) & 0x7fffffff, __double2hiint(v[c].im) & 0x7fffffff));
                if (e < 0x100000) {  // zeros, or subnormal numbers, which have no fixed-point form here
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (v[c].re != 0.0 || v[c].im != 0.0) ok = false;
                    continue;
                }
                e >>= 20;
                if (e > E) {
                    // the unit follows the largest neighbour so far; the first one takes a binade of
                    // headroom, so that later ones seldom move it
                    const int en = E == 0 ? e + 1 : e;
                    if (E != 0) {
#pragma unroll
                        for (int r = 0; r < 3; ++r)
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                hh[r][q] = fx_shift(hh[r][q], en - E);
                                mid[r][q] = fx_shift(mid[r][q], en - E);
                            }
                    }
                    E = en;
                }
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const FxNum xr = fx_limbs(flip ? -v[c].re : v[c].re, E);
                    const FxNum xi = fx_limbs(flip ? -v[c].im : v[c].im, E);
                    const FxNum n = fx_neg(back ? xr : xi);
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const FxNum &re = back ? u[c][r][0] : u[r][c][0], &im = back ? u[c][r][1] : u[r][c][1];
                        fx_mac(hh[r][0], mid[r][0], re, xr);
                        fx_mac(hh[r][0], mid[r][0], im, back ? xi : n);
                        fx_mac(hh[r][1], mid[r][1], re, xi);
                        fx_mac(hh[r][1], mid[r][1], im, back ? n : xr);
                    }
                }
            }
        }
        ok &= E == 0 || (E >= 100 && E < 2046);
        if (ok) {
            const double unit = __hiloint2double(max(E - 54, 0) << 20, 0);  // of hh: 2^56 2^(E - 1078) 2^-55
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                acc[0][r].re = unit * (double)(hh[r][0] + ((mid[r][0] + (1 << 27)) >> 28));
                acc[0][r].im = unit * (double)(hh[r][1] + ((mid[r][1] + (1 << 27)) >> 28));
            }
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[0][c] = cx<double>{0.0, 0.0};
#pragma unroll 1
            for (int mu = 0; mu < 4; ++mu) {
                const Hop hp = hop_of(G.g, s, mu);
                cx<double> U[3][3], v[3];
                LinkF64R18::load(link_block<LinkF64R18>(G.links, Vh, mu, op), Vh, h, U);
                Field<double>::load(G.in[0], Vh, hp.hf, v);
                dp_hop<false>(acc[0], U, v, hp.sf);
                LinkF64R18::load(link_block<LinkF64R18>(G.links, Vh, mu, 1 - op), Vh, hp.hb, U);
                Field<double>::load(G.in[0], Vh, hp.hb, v);
                dp_hop<true>(acc[0], U, v, -hp.sb);
            }
        }
    }

    const bool act[1] = {true};
    __shared__ double sh[32];
    dslash_epilogue<double, 1, MODE, BS>(G, bx, act, live, h, acc, sh);
}

// Small lattices (up to kFxSplitVh sites per parity): a block covers 64 output sites with four threads
// each.  Thread (mu, site) does the two hops of one direction, so that every load of a site is in
// flight at once and few sites fill the chip; the four partial sums meet in shared memory in the unit
// of the largest neighbour.  One right-hand side, against one thread per site: 12^4 13.6 -> 9.2 us, 16^4
// 22.5 -> 14.8 us, 20^4 34.7 -> 30.4 us, but 24^4 56.4 -> 57.3 us (normal operator 122 -> 128 us) and 32^4
// 151 -> 168 us, where the exchange costs more than the parallelism gives.  The choice depends on
// the lattice alone, so that results do not depend on what else a launch carries.
constexpr int kFxSites = 64;
constexpr int kFxSplitVh = 90000;

template <int MODE>
__global__ void __launch_bounds__(4 * kFxSites, 3) k_dslash_fx4(const __grid_constant__ DArgs a)
{
    pdl_enter();
    const int bx = block_along_sites();
    const DGroup &G = a.grp[blockIdx.x];
    const int Vh = G.g.Vh;
    if (bx * kFxSites >= G.g.h_end - G.g.h_begin) return;             // block-uniform
    if (G.nrhs < 1 || (G.skip[0] != nullptr && *G.skip[0] != 0)) return;  // block-uniform

    __shared__ long long s_part[3][12][kFxSites];  // sums of mu = 1..3 (as doubles on the FP64 path)
    __shared__ int s_e[4][kFxSites];               // exponent of each sum's unit; -1: no fixed-point form
    __shared__ double sh[32];
    const int mu = threadIdx.x / kFxSites, sl = threadIdx.x % kFxSites;  // mu is warp-uniform
    const int h = G.g.h_begin + bx * kFxSites + sl;
    const bool live = h < G.g.h_end;
    const int op = a.out_par;
    Hop hp;
    if (live) hp = hop_of(G.g, site_of(G.g, op, h), mu);

    long long hh[3][2], mid[3][2];
#pragma unroll
    for (int r = 0; r < 3; ++r) hh[r][0] = hh[r][1] = mid[r][0] = mid[r][1] = 0;
    int E = 0;  // 0 while both neighbours are zero
    if (live) {
        cx<double> v[2][3];
        Field<double>::load(G.in[0], Vh, hp.hf, v[0]);
        Field<double>::load(G.in[0], Vh, hp.hb, v[1]);
        bool ok = *G.fx_bad == 0;
        int e = 0, tiny = 0;
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c)
                e = max(e, max(__double2hiint(v[k][c].re) & 0x7fffffff, __double2hiint(v[k][c].im) & 0x7fffffff));
        E = e >> 20;
        if (E == 0) {  // zeros, or subnormal numbers, which have no fixed-point form here
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int c = 0; c < 3; ++c) tiny |= v[k][c].re != 0.0 || v[k][c].im != 0.0;
        }
        ok = ok && !tiny && (E == 0 || (E >= 100 && E < 2046));
        if (E != 0) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool back = k == 1;
                const bool flip = back ? hp.sb > 0.f : hp.sf < 0.f;  // the backward hop enters with -u
                FxNum u[3][3][2];
                LinkFX::load(link_block<LinkFX>(G.fx_links, Vh, mu, back ? 1 - op : op), Vh, back ? hp.hb : h, u);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const FxNum xr = fx_limbs(flip ? -v[k][c].re : v[k][c].re, E);
                    const FxNum xi = fx_limbs(flip ? -v[k][c].im : v[k][c].im, E);
                    const FxNum n = fx_neg(back ? xr : xi);
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const FxNum &re = back ? u[c][r][0] : u[r][c][0], &im = back ? u[c][r][1] : u[r][c][1];
                        fx_mac(hh[r][0], mid[r][0], re, xr);
                        fx_mac(hh[r][0], mid[r][0], im, back ? xi : n);
                        fx_mac(hh[r][1], mid[r][1], re, xi);
                        fx_mac(hh[r][1], mid[r][1], im, back ? n : xr);
                    }
                }
            }
        }
        s_e[mu][sl] = ok ? E : -1;
        if (!ok) E = -1;
        if (mu > 0) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    s_part[mu - 1][4 * r + 2 * q][sl] = hh[r][q];
                    s_part[mu - 1][4 * r + 2 * q + 1][sl] = mid[r][q];
                }
        }
    }
    cx<double> acc[1][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[0][c] = cx<double>{0.0, 0.0};
    const bool any_bad = __syncthreads_or(E < 0);
    const bool bad = any_bad && live && min(min(s_e[0][sl], s_e[1][sl]), min(s_e[2][sl], s_e[3][sl])) < 0;
    if (any_bad) {
        if (bad) {  // this direction in FP64
            cx<double> U[3][3], v[3];
            LinkF64R18::load(link_block<LinkF64R18>(G.links, Vh, mu, op), Vh, h, U);
            Field<double>::load(G.in[0], Vh, hp.hf, v);
            dp_hop<false>(acc[0], U, v, hp.sf);
            LinkF64R18::load(link_block<LinkF64R18>(G.links, Vh, mu, 1 - op), Vh, hp.hb, U);
            Field<double>::load(G.in[0], Vh, hp.hb, v);
            dp_hop<true>(acc[0], U, v, -hp.sb);
            if (mu > 0)
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    s_part[mu - 1][2 * r][sl] = __double_as_longlong(acc[0][r].re);
                    s_part[mu - 1][2 * r + 1][sl] = __double_as_longlong(acc[0][r].im);
                }
        }
        __syncthreads();
    }
    if (live && mu == 0) {
        if (bad) {
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    acc[0][r].re += __longlong_as_double(s_part[m][2 * r][sl]);
                    acc[0][r].im += __longlong_as_double(s_part[m][2 * r + 1][sl]);
                }
        } else {
            const int em[4] = {E, s_e[1][sl], s_e[2][sl], s_e[3][sl]};
            const int top = max(max(em[0], em[1]), max(em[2], em[3]));
            const double unit = __hiloint2double(max(top - 54, 0) << 20, 0);  // of hh: 2^56 2^(top - 1078) 2^-55
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    long long sum = fx_shift(hh[r][q], top - em[0]), low = fx_shift(mid[r][q], top - em[0]);
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        sum += fx_shift(s_part[m][4 * r + 2 * q][sl], top - em[m + 1]);
                        low += fx_shift(s_part[m][4 * r + 2 * q + 1][sl], top - em[m + 1]);
                    }
                    const double w = unit * (double)(sum + ((low + (1 << 27)) >> 28));
                    if (q == 0)
                        acc[0][r].re = w;
                    else
                        acc[0][r].im = w;
                }
        }
    }
    const bool act[1] = {true};
    dslash_epilogue<double, 1, MODE, kFxSites>(G, bx, act, live && mu == 0, h, acc, sh);
}

}  // namespace stg
