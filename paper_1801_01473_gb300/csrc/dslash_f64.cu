// D_eo / D_oe instantiations for FP64 links (18-real and 12-real) on FP64 fields.
#include <cstring>

#include "dslash_fx.cuh"
#include "stg_common.h"

namespace stg {

template <int BS>
static cudaError_t launch_fx_b(const DArgs &a, int mode, int maxv, cudaStream_t st)
{
    if (mode == 0) return launch_sites(k_dslash_fx<0, BS>, maxv, BS, BS, 0, st, a);
    if (mode == 1) return launch_sites(k_dslash_fx<1, BS>, maxv, BS, BS, 0, st, a);
    return launch_sites(k_dslash_fx<2, BS>, maxv, BS, BS, 0, st, a);
}

static cudaError_t launch_fx4(const DArgs &a, int mode, int maxv, cudaStream_t st)
{
    if (mode == 0) return launch_sites(k_dslash_fx4<0>, maxv, kFxSites, 4 * kFxSites, 0, st, a);
    if (mode == 1) return launch_sites(k_dslash_fx4<1>, maxv, kFxSites, 4 * kFxSites, 0, st, a);
    return launch_sites(k_dslash_fx4<2>, maxv, kFxSites, 4 * kFxSites, 0, st, a);
}

cudaError_t launch_dslash_f64r18(const DArgs &a, int mode, int bs, cudaStream_t st)
{
    int maxv, maxr;
    dslash_extent(a, maxv, maxr);
    if (a.ngroups <= 0 || maxv <= 0 || maxr <= 0) return cudaSuccess;
    // launch_dslash splits the groups of fixed-point links to one right-hand side
    bool fx = maxr == 1;
    for (int k = 0; k < a.ngroups; ++k) fx = fx && a.grp[k].fx_links;
    if (!fx) return launch_dslash_t<LinkF64R18>(a, mode, bs, st);
    // small lattices by four threads per site; a launch with both kinds becomes two
    int nsplit = 0;
    for (int k = 0; k < a.ngroups; ++k) nsplit += a.grp[k].g.Vh <= kFxSplitVh;
    if (nsplit == a.ngroups) return launch_fx4(a, mode, maxv, st);
    if (nsplit > 0) {
        for (int split = 0; split < 2; ++split) {
            DArgs b;
            memset(&b, 0, sizeof(b));
            b.out_par = a.out_par;
            for (int k = 0; k < a.ngroups; ++k)
                if ((a.grp[k].g.Vh <= kFxSplitVh) == (split == 1)) b.grp[b.ngroups++] = a.grp[k];
            const cudaError_t e = launch_dslash_f64r18(b, mode, bs, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    if (bs == 64) return launch_fx_b<64>(a, mode, maxv, st);
    if (bs == 256) return launch_fx_b<256>(a, mode, maxv, st);
    return launch_fx_b<128>(a, mode, maxv, st);
}
cudaError_t launch_dslash_f64r12(const DArgs &a, int mode, int bs, cudaStream_t st) { return launch_dslash_t<LinkF64R12>(a, mode, bs, st); }

// The state beside a fixed-point copy before its links are written: no link without the form yet, and the
// exponent of the links' unit, the power of two at or above the first link's |U| / sqrt 3 (1 for SU(3)).
__global__ void k_fx_begin(const double2 *__restrict__ first, int *state)
{
    double n = 0.0;
    for (int k = 0; k < 9; ++k) {
        const double2 u = first[k];
        n = fma(u.x, u.x, fma(u.y, u.y, n));
    }
    n = sqrt(n / 3.0) * (1.0 - 0x1p-20);
    int ke = 0;
    if (n > 0x1p-400 && n < 0x1p400) {
        const int hi = __double2hiint(n);
        ke = (hi >> 20) - 1023 + ((hi & 0xfffff) != 0 || __double2loint(n) != 0 ? 1 : 0);
    }
    state[0] = 0;
    state[1] = ke;
}

// One thread per link (mu, i), as k_pack_links; state[0] is set when some link has no fixed-point form.
// Bound by HBM (a link read once and written twice): update of a 32^4 gauge 294 us, links alone 210.
__global__ void k_pack_links_fx(Geom g, const double2 *__restrict__ canon, void *__restrict__ links,
                                void *__restrict__ fx_links, int *state)
{
    const long long V = 2LL * g.Vh, tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= 4 * V) return;
    const int mu = (int)(tid / V), i = (int)(tid - mu * V), ke = state[1];
    const int x = i % g.L[0], r = i / g.L[0], y = r % g.L[1], r2 = r / g.L[1], z = r2 % g.L[2], t = r2 / g.L[2];
    double2 m[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) m[k] = canon[tid * 9 + k];
    const size_t blk = (size_t)(mu * 2 + ((x + y + z + t) & 1)) * g.Vh * LinkF64R18::kBytes;
    LinkF64R18::pack(static_cast<char *>(links) + blk, g.Vh, i >> 1, m);
    if (!LinkFX::pack(static_cast<char *>(fx_links) + blk, g.Vh, i >> 1, m, ke)) state[0] = 1;
}

cudaError_t launch_pack_links_fx(const Geom &g, const void *canon, void *links, void *fx_links, int *state,
                                 cudaStream_t st)
{
    static_assert(LinkFX::kBytes == LinkF64R18::kBytes, "the copy has the size and the blocks of the links");
    const double2 *c = static_cast<const double2 *>(canon);
    k_fx_begin<<<1, 1, 0, st>>>(c, state);
    k_pack_links_fx<<<(unsigned)((8LL * g.Vh + 255) / 256), 256, 0, st>>>(g, c, links, fx_links, state);
    return cudaGetLastError();
}
}  // namespace stg
