// dslash_fx.cuh -- the hopping term on FP64 18-real links with its products on the integer pipes.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM, so the 288 products of an output site bind
// the FP64 operator at a third of the memory bandwidth.  The integer pipes multiply 32 x 32 -> 64 bits
// with a 64-bit accumulator at ~30 per clock and SM (measured), so three of those per product are
// faster.  Links (entries up to a power of two, here 1, in units of 2^-57 of it) and the neighbour vectors
// of a site (unit 2^-58 of B, a power of two above the largest of them) are signed fixed-point numbers in
// two limbs,
// value = l1 2^29 + l0 with |l0| <= 2^28, |l1| <= 2^28 (links) or 2^29 (vectors), and
//   sum u v = 2^58 sum u1 v1 + 2^29 sum (u1 v0 + u0 v1)      (u0 v0 is dropped)
// with both sums exact in 64 bits: the real numbers of a link's row or column add up to at most 2.5 (pack;
// sqrt 6 for unitary links), so that the first is at most 20 * 2^57 and the second 20 * 2^56 + 48 * 2^57.
//
// Where it may be used.  A component's error is at most ~2^-52.9 B (48 dropped products of 2^-59 B, 48
// vector numbers rounded by 2^-59 B), ~2^-57.3 B rms, whatever the component's own size, where an FP64 sum
// lies within 14 * 2^-53 of sum |u||v| (6 roundings a hop, 8 additions), 0.45 * 2^-53 rms.  So every real
// component must have sum |u||v| >= 5/64 B, which makes the first bound no larger than the second.
// A lower bound of sum |u||v| comes with the sums: the absolute contributions of the eight hops, from the
// accumulators' high words (all of it costs 3 % of the kernel).  With Gaussian vectors and mixing links it is
// ~1.4 B, and below 5/64 B for less than 1e-5 of the sites.  What fails (small links, colours and parts that
// links do not mix with larger ones, point sources) goes through FP64 site by site.  So do infinities,
// NaNs, subnormal numbers and vectors near the ends of the exponent range, and whole gauges with a
// link whose largest entry is outside [2^-4, 1] (zero links are fine) or that fails the 2.5.  The power of
// two is the one at or above the first link's size (k_fx_begin), so that scaled links keep the fixed point.
//
// D back to back, FP64 kernel -> this: 32^4 312 -> 154 us (of 100 us at the copy bandwidth), 24^4 108 ->
// 57 us, 16^4 36 -> 14 us, 8^4 14 -> 6 us; a gauge without fixed-point form 32^4 339, 24^4 116, 16^4 28 us, real
// fields on unit links (no imaginary part to find) 356, 124, 34 us.  What bounds it: the integer pipes (864 products and ~1500
// other operations a site) and, with one thread per site, loads in flight at 16 to 20 warps per SM.
#pragma once

#include "dslash.cuh"

namespace stg {

struct FxNum {
    int l1, l0;
};

constexpr int kFxLow = 29;  // bits of the low limb

// limbs of w / 2, rounded.  The high limb is rounded too: the low one is balanced around zero.
__device__ __forceinline__ FxNum fx_split_half(long long w)
{
    w += (1 << kFxLow) + 1;
    FxNum r;
    r.l1 = (int)(w >> (kFxLow + 1));
    r.l0 = (int)(((unsigned)w >> 1) & ((1u << kFxLow) - 1)) - (1 << (kFxLow - 1));
    return r;
}

// d in units of 2^(E - 1080), rounded, for |d| < 2^(E - 1022) = B (E a biased exponent)
__device__ __forceinline__ FxNum fx_limbs(double d, int E)
{
    const int hi = __double2hiint(d);
    const unsigned lo = (unsigned)__double2loint(d);
    // (E << 20 | 0xfffff) - |hi| has E - e in its top bits (e the exponent of d)
    const int k = ((E << 20 | 0xfffff) - (hi & 0x7fffffff)) >> 20;
    const unsigned mh = (__funnelshift_l(lo, (unsigned)hi, 10) & 0x3fffffffu) | 0x40000000u;  // significand from bit 62
    const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 10);
    const long long v = (long long)(m >> min(k + 4, 63));
    const long long sg = (long long)(hi >> 31);
    return fx_split_half((v ^ sg) - sg);
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

// The high word of a sum of u1 v1 is in units of 2^-25 B.
constexpr unsigned kFxLeast = 5u << 19;   // 5/64 B, of a whole component
constexpr unsigned kFxLeast2 = 1u << 13;  // 2^-12 B, of the two hops of one direction: random numbers hardly ever
__device__ __forceinline__ int fx_high(long long hh) { return (int)(hh >> 32); }
__device__ __forceinline__ unsigned fx_min(const unsigned size[3][2])
{
    return min(min(min(size[0][0], size[0][1]), min(size[1][0], size[1][1])), min(size[2][0], size[2][1]));
}

// d 2^(58 - ke) rounded, |d| < 2^(ke + 1), on the integer pipes: in FP64 the copy of a gauge was bound by
// the multiplications and conversions
__device__ __forceinline__ long long fx_round58(double d, int ke)
{
    const int hi = __double2hiint(d);
    const int e = ((hi & 0x7fffffff) >> 20) - ke;  // d = significand 2^(e + ke - 1075)
    const long long m = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(d);
    const int s = 1017 - e;  // significand 2^(e - 1075 + 58)
    const long long v = s <= 0 ? m << -s : fx_shift(m, s);  // s >= -6: below 2^59
    return hi < 0 ? -v : v;
}

// |d| in units of 2^(ke - 20), truncated, from its high word (|d| < 2^(ke + 1); others give some finite number)
__device__ __forceinline__ float fx_unit20(int hi, int ke)
{
    return (float)(((hi & 0xfffff) | 0x100000) >> min(max(1023 + ke - (hi >> 20), 0), 31));
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
    // ke: exponent of the unit.  False when the link has no fixed-point form: an entry above 1 or a row or
    // column of more than 2.5 (by more than the hair's breadth that rounding takes a unitary matrix past
    // it), or all entries of a link that is not zero below 2^-4, in that unit
    __device__ __forceinline__ static bool pack(void *blk, int Vh, int h, const double2 *m, int ke)
    {
        int4 *p = static_cast<int4 *>(blk);
        int top = 0, any = 0;
        float row[3] = {0.f, 0.f, 0.f}, col[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int re = __double2hiint(m[k].x) & 0x7fffffff, im = __double2hiint(m[k].y) & 0x7fffffff;
            top = max(top, max(re, im));
            any |= re | im | __double2loint(m[k].x) | __double2loint(m[k].y);
            // entries of at most 1 (top), in units of 2^-20 from the bits of the significand
            const float sum = fx_unit20(re, ke) + fx_unit20(im, ke);
            row[k / 3] += sum;
            col[k % 3] += sum;
        }
        const float most = fmaxf(fmaxf(fmaxf(row[0], row[1]), row[2]), fmaxf(fmaxf(col[0], col[1]), col[2]));
        const int one = 0x3ff00000 + ke * (1 << 20), sixteenth = one - 0x00400000;
        const bool ok = top <= one && (any == 0 || top >= sixteenth) && most <= 2.4999f * (1 << 20);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const FxNum re = fx_split_half(ok ? fx_round58(m[k].x, ke) : 0);
            const FxNum im = fx_split_half(ok ? fx_round58(m[k].y, ke) : 0);
            p[(size_t)k * Vh + h] = make_int4(re.l1, re.l0, im.l1, im.l0);
        }
        return ok;
    }
};

// ---- sites in FP64.  Three forms with one order of summation, so that a site's value does not depend on its
// neighbours in the warp: the 6 terms of a direction, then (x + y) + (z + t).

// acc = the two hops of direction mu
__device__ __forceinline__ void dp_direction(const DGroup &G, int op, int h, int mu, const Hop &hp, cx<double> acc[3])
{
    const int Vh = G.g.Vh;
#pragma unroll
    for (int r = 0; r < 3; ++r) acc[r] = cx<double>{0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool back = k == 1;
        cx<double> U[3][3], v[3];
        LinkF64R18::load(link_block<LinkF64R18>(G.links, Vh, mu, back ? 1 - op : op), Vh, back ? hp.hb : h, U);
        Field<double>::load(G.in[0], Vh, back ? hp.hb : hp.hf, v);
        if (back ? hp.sb > 0.f : hp.sf < 0.f) neg3(v);  // the backward hop enters with -u
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (back)
                    cmac_conj(acc[r], U[c][r], v[c]);
                else
                    cmac(acc[r], U[r][c], v[c]);
            }
    }
}

__device__ __forceinline__ void dp_add(cx<double> a[3], const cx<double> b[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c] = cx<double>{a[c].re + b[c].re, a[c].im + b[c].im};
}

// The sites of the lanes with `need`, for a whole warp.  A few of them (kDpLanes) are taken one by one with a lane
// per direction and row: a warp holds the FP64 pipe for 64 cycles an instruction, so a lane that does its
// site's 288 multiply-adds alone takes ~10 us, which a launch of a small lattice has to wait for.
constexpr int kDpLanes = 8;
__device__ __forceinline__ void dp_sites(const DGroup &G, int op, int h, bool need, cx<double> acc[3])
{
    unsigned todo = __ballot_sync(0xffffffffu, need);
    if (todo == 0) return;
    if (__popc(todo) > kDpLanes) {
        if (!need) return;
        const Site s = site_of(G.g, op, h);
#pragma unroll 1
        for (int pair = 0; pair < 2; ++pair) {
            cx<double> a[3], b[3];
            dp_direction(G, op, h, 2 * pair, hop_of(G.g, s, 2 * pair), a);
            dp_direction(G, op, h, 2 * pair + 1, hop_of(G.g, s, 2 * pair + 1), b);
            dp_add(a, b);
            if (pair == 0) {
#pragma unroll
                for (int c = 0; c < 3; ++c) acc[c] = a[c];
            } else {
                dp_add(acc, a);
            }
        }
        return;
    }
    const int Vh = G.g.Vh, lane = threadIdx.x & 31;
    const int r = lane >> 2, mu = lane & 3;
#pragma unroll 1
    while (todo != 0) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int hs = __shfl_sync(0xffffffffu, h, src);
        cx<double> w = cx<double>{0.0, 0.0};
        if (r < 3) {
            const Hop hp = hop_of(G.g, site_of(G.g, op, hs), mu);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool back = k == 1;
                const double2 *U = static_cast<const double2 *>(link_block<LinkF64R18>(G.links, Vh, mu, back ? 1 - op : op));
                cx<double> v[3];
                Field<double>::load(G.in[0], Vh, back ? hp.hb : hp.hf, v);
                if (back ? hp.sb > 0.f : hp.sf < 0.f) neg3(v);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double2 e = __ldg(U + (size_t)(back ? 3 * c + r : 3 * r + c) * Vh + (back ? hp.hb : hs));
                    if (back)
                        cmac_conj(w, cx<double>{e.x, e.y}, v[c]);
                    else
                        cmac(w, cx<double>{e.x, e.y}, v[c]);
                }
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            w.re += __shfl_xor_sync(0xffffffffu, w.re, o);
            w.im += __shfl_xor_sync(0xffffffffu, w.im, o);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cx<double> t = cx<double>{__shfl_sync(0xffffffffu, w.re, 4 * c), __shfl_sync(0xffffffffu, w.im, 4 * c)};
            if (lane == src) acc[c] = t;
        }
    }
}

// One thread per output site.  Blocks of 128 threads are held to 96 registers with a few spills (five
// blocks per SM: 24^4 58.7 -> 57.0 us), blocks of 64 and 256 keep 128.
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
    bool ok = true;

    if (live) {
        const Site s = site_of(G.g, op, h);
        long long hh[3][2], mid[3][2];
        int E = 0;  // exponent of the unit's power of two; 0 while all neighbours were zero
        ok = G.fx_state[0] == 0;
        const int ke = G.fx_state[1];
        unsigned size[3][2];  // lower bounds of sum |u||v|
#pragma unroll
        for (int r = 0; r < 3; ++r) hh[r][0] = hh[r][1] = mid[r][0] = mid[r][1] = size[r][0] = size[r][1] = 0;
        // one direction per turn: all four unrolled are ~64 KB of instructions and ran slower
#pragma unroll 1
        for (int mu = ok ? 0 : 4; mu < 4; ++mu) {
            const Hop hp = hop_of(G.g, s, mu);
            int before[3][2];  // high words of hh before the hop
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) before[r][q] = fx_high(hh[r][q]);
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
                    const int en = E == 0 ? min(e + 1, 2047) : e;
                    if (E != 0) {
#pragma unroll
                        for (int r = 0; r < 3; ++r)
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                hh[r][q] = fx_shift(hh[r][q], en - E);
                                mid[r][q] = fx_shift(mid[r][q], min(en - E, 60));  // room for the rounding
                                size[r][q] >>= min(en - E, 31);
                                before[r][q] >>= min(en - E, 31);
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
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        size[r][q] = __sad(fx_high(hh[r][q]), before[r][q], size[r][q]);
                        before[r][q] = fx_high(hh[r][q]);
                    }
            }
            // what the first direction already shows (links that do not mix) costs only that
            if (mu == 0 && E != 0 && fx_min(size) < kFxLeast2) {
                ok = false;
                break;
            }
        }
        ok = ok && (E == 0 || (E >= 100 && E < 2046 && E + ke >= 100 && E + ke < 2046 && fx_min(size) >= kFxLeast));
        if (ok) {
            const double unit = __hiloint2double(max(E + ke - 56, 0) << 20, 0);  // of hh: 2^58 2^(E - 1080) 2^(ke - 57)
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                acc[0][r].re = unit * (double)(hh[r][0] + ((mid[r][0] + (1 << (kFxLow - 1))) >> kFxLow));
                acc[0][r].im = unit * (double)(hh[r][1] + ((mid[r][1] + (1 << (kFxLow - 1))) >> kFxLow));
            }
        }
    }
    dp_sites(G, op, h, !ok, acc[0]);

    const bool act[1] = {true};
    __shared__ double sh[32];
    dslash_epilogue<double, 1, MODE, BS>(G, bx, act, live, h, acc, sh);
}

// Small lattices (up to kFxSplitVh sites per parity): a block covers 64 output sites with four threads
// each.  Thread (mu, site) does the two hops of one direction, so that every load of a site is in
// flight at once and few sites fill the chip; the four partial sums meet in shared memory in the unit
// of the largest neighbour.  Back to back, one thread per site -> four: D 8^4 11.5 -> 6.0 us, 12^4 12.5 -> 10.3, 16^4 20.7
// -> 14.0, 20^4 34.1 -> 30.1, but 24^4 57.5 -> 59.9 (normal operator 123 -> 130 us) and 32^4 155 -> 165, where the
// exchange costs more than the parallelism gives.  The choice depends on the lattice alone, so that
// results do not depend on what else a launch carries.
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
    __shared__ unsigned s_size[3][6][kFxSites];    // lower bounds of sum |u||v| of mu = 1..3
    __shared__ double sh[32];
    const int mu = threadIdx.x / kFxSites, sl = threadIdx.x % kFxSites;  // mu is warp-uniform
    const int h = G.g.h_begin + bx * kFxSites + sl;
    const bool live = h < G.g.h_end;
    const int op = a.out_par;
    const int ke = G.fx_state[1];
    Hop hp;
    if (live) hp = hop_of(G.g, site_of(G.g, op, h), mu);

    long long hh[3][2], mid[3][2];
#pragma unroll
    for (int r = 0; r < 3; ++r) hh[r][0] = hh[r][1] = mid[r][0] = mid[r][1] = 0;
    unsigned size[3][2] = {{0, 0}, {0, 0}, {0, 0}};
    int E = 0;  // 0 while both neighbours are zero
    if (live) {
        cx<double> v[2][3];
        Field<double>::load(G.in[0], Vh, hp.hf, v[0]);
        Field<double>::load(G.in[0], Vh, hp.hb, v[1]);
        bool ok = G.fx_state[0] == 0;
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
        ok = ok && !tiny && (E == 0 || (E >= 100 && E < 2046 && E + ke >= 100 && E + ke < 2046));
        if (E != 0 && ok) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const bool back = k == 1;
                const bool flip = back ? hp.sb > 0.f : hp.sf < 0.f;  // the backward hop enters with -u
                FxNum u[3][3][2];
                LinkFX::load(link_block<LinkFX>(G.fx_links, Vh, mu, back ? 1 - op : op), Vh, back ? hp.hb : h, u);
                int before[3][2];
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int q = 0; q < 2; ++q) before[r][q] = fx_high(hh[r][q]);
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
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int q = 0; q < 2; ++q) size[r][q] = __sad(fx_high(hh[r][q]), before[r][q], size[r][q]);
            }
            ok = fx_min(size) >= kFxLeast2;  // links that do not mix
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
                    s_size[mu - 1][2 * r + q][sl] = size[r][q];
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
            dp_direction(G, op, h, mu, hp, acc[0]);
            if (mu > 0)
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    s_part[mu - 1][2 * r][sl] = __double_as_longlong(acc[0][r].re);
                    s_part[mu - 1][2 * r + 1][sl] = __double_as_longlong(acc[0][r].im);
                }
        }
        __syncthreads();
    }
    if (mu == 0) {
        bool need = false;
        if (bad) {
            cx<double> x[3][3];
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    x[m][r] = cx<double>{__longlong_as_double(s_part[m][2 * r][sl]),
                                         __longlong_as_double(s_part[m][2 * r + 1][sl])};
            dp_add(acc[0], x[0]);
            dp_add(x[1], x[2]);
            dp_add(acc[0], x[1]);
        } else if (live) {
            const int em[4] = {E, s_e[1][sl], s_e[2][sl], s_e[3][sl]};
            const int top = max(max(em[0], em[1]), max(em[2], em[3]));
            const double unit = __hiloint2double(max(top + ke - 56, 0) << 20, 0);  // of hh: 2^58 2^(top - 1080) 2^(ke - 57)
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    size[r][q] >>= min(top - em[0], 31);
#pragma unroll
                    for (int m = 0; m < 3; ++m) size[r][q] += s_size[m][2 * r + q][sl] >> min(top - em[m + 1], 31);
                    long long sum = fx_shift(hh[r][q], top - em[0]), low = fx_shift(mid[r][q], top - em[0]);
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        sum += fx_shift(s_part[m][4 * r + 2 * q][sl], top - em[m + 1]);
                        low += fx_shift(s_part[m][4 * r + 2 * q + 1][sl], top - em[m + 1]);
                    }
                    const double w = unit * (double)(sum + ((low + (1 << (kFxLow - 1))) >> kFxLow));
                    if (q == 0)
                        acc[0][r].re = w;
                    else
                        acc[0][r].im = w;
                }
            need = top != 0 && fx_min(size) < kFxLeast;
        }
        dp_sites(G, op, h, need, acc[0]);
    }
    const bool act[1] = {true};
    dslash_epilogue<double, 1, MODE, kFxSites>(G, bx, act, live && mu == 0, h, acc, sh);
}

}  // namespace stg
