"""The FP64 operator's fixed-point kernels (k_dslash_fx, k_dslash_fx4) against the FP64 oracle, and the sites that it
hands to its FP64 loop: components of very different size at neighbouring sites and within a site,
zero neighbourhoods, the ends of the exponent range, infinities and NaNs, links of 2 and above; one
and several right-hand sides, the smallest lattice that takes it (2048 sites), one below it, extents
of 2 and remainders of the thread block.

Tolerance: fixed-point numbers carry 2^-55 of the largest neighbour component, the dropped low
products and 48 terms keep the sum below 2^-50 of it; 1e-14 of the largest input in a site's
neighbourhood (links of order one) therefore bounds the error of that site.
"""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu

LARGE = (24, 24, 24, 14)  # 96768 sites per parity: one thread per site (four below 90000)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _neighbour_max(dims, psi, out_par):
    """Largest |component| among the 8 neighbours of every site of parity out_par."""
    v = int(np.prod(dims))
    x = np.stack(np.unravel_index(np.arange(v), dims[::-1])[::-1])
    par = x.sum(0) % 2
    full = np.zeros(v)
    comp = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(-1)
    full[par != out_par] = comp
    grid = full.reshape(dims[::-1])
    near = np.max([np.roll(grid, s, axis=a) for a in range(4) for s in (1, -1)], axis=0).reshape(-1)
    return near[par == out_par]


def _check(dims, u, psi, factor=1.0):
    import paper_1801_01473_gb300 as p
    g = p.Gauge(p.Lattice(dims), _gpu(u), "f64", 18)
    for par, ref in ((1, oracle.dslash_oe), (0, oracle.dslash_eo)):
        got = p.dslash(g, par, _gpu(psi)).cpu().numpy()
        want = ref(dims, u, psi)
        bound = 1e-14 * factor * _neighbour_max(dims, psi, par)[:, None]
        assert (np.abs(got - want) <= bound).all()


@pytest.mark.parametrize("dims", [(8, 8, 8, 4), (2, 2, 32, 16), (6, 10, 4, 14), (4, 4, 4, 4), LARGE])
def test_matches_oracle(dims):
    _check(dims, S.gauge_links(dims, "haar", 171), S.gaussian_field(dims, 172))


@pytest.mark.parametrize("dims", [(8, 6, 6, 8), LARGE])
@pytest.mark.parametrize("scale", [1e-290, 1e-30, 1e30, 1e290])
def test_scales(scale, dims):
    """Vectors far from one, and (1e-290) below the exponents that the fixed-point form takes."""
    _check(dims, S.gauge_links(dims, "haar", 173), scale * S.gaussian_field(dims, 174))


@pytest.mark.parametrize("dims", [(8, 6, 8, 6), LARGE])
def test_uneven_sizes_and_zeros(dims):
    """Sizes spread over 60 decades site by site and colour by colour, with zeros and zero sites."""
    rng = np.random.default_rng(175)
    psi = S.gaussian_field(dims, 176)
    psi = psi * 10.0 ** rng.uniform(-60, 0, psi.shape[:1])[:, None] * 10.0 ** rng.uniform(-8, 0, psi.shape)
    psi[rng.random(psi.shape[0]) < 0.6] = 0.0
    psi[rng.random(psi.shape) < 0.2] = 0.0
    _check(dims, S.gauge_links(dims, "haar", 177), psi)
    point = np.zeros_like(psi)
    point[3, 1] = 1.0 - 2.0j
    _check(dims, S.gauge_links(dims, "haar", 177), point)


@pytest.mark.parametrize("dims", [(4, 8, 8, 8), LARGE])
def test_links_outside_the_fixed_point_range(dims):
    u = S.gauge_links(dims, "haar", 178).copy()
    u[2, 17] *= 1e3
    _check(dims, u, S.gaussian_field(dims, 179), factor=1e3)


@pytest.mark.parametrize("dims", [(8, 6, 8, 8), LARGE])
def test_non_finite_inputs_stay_local(dims):
    """Sites with a NaN or infinite neighbour are not finite, as in the FP64 loop; the others are the same."""
    import paper_1801_01473_gb300 as p
    u = S.gauge_links(dims, "haar", 180)
    psi = S.gaussian_field(dims, 181)
    g = p.Gauge(p.Lattice(dims), _gpu(u), "f64", 18)
    for bad in (np.nan, np.inf):
        broken = psi.copy()
        broken[5, 2] = bad
        want = oracle.dslash_oe(dims, u, broken)
        got = p.dslash(g, 1, _gpu(broken)).cpu().numpy()
        finite = np.isfinite(want).all(-1)
        assert (~finite).any() and (np.isfinite(got).all(-1) == finite).all()
        assert np.abs(got[finite] - want[finite]).max() <= 1e-13


@pytest.mark.parametrize("nrhs", [2, 19])
def test_several_right_hand_sides_and_update(nrhs):
    """Bitwise the single results, also after the gauge has taken new links."""
    import paper_1801_01473_gb300 as p
    dims = (8, 6, 8, 6)
    lat = p.Lattice(dims)
    g = p.Gauge(lat, _gpu(S.gauge_links(dims, "haar", 182)), "f64", 18)
    psi = [S.gaussian_field(dims, 183 + j) for j in range(nrhs)]
    p.dslash(g, 0, _gpu(psi[0]))
    u = S.gauge_links(dims, "haar", 184)
    g.update(_gpu(u))
    inp = torch.stack([p.pack(lat, _gpu(s), "f64") for s in psi])
    out = torch.empty_like(inp)
    p.dslash_multi_(g, 0, out, inp)
    for j in range(nrhs):
        assert torch.equal(out[j], p.dslash_eo_(g, torch.empty_like(inp[j]), inp[j].contiguous()))
    want = oracle.dslash_eo(dims, u, psi[nrhs - 1])
    assert np.abs(p.unpack(lat, out[nrhs - 1]).cpu().numpy() - want).max() <= 1e-13


def test_lattices_of_both_kinds_in_one_batch():
    """A batched FP64 solve over a lattice of each kernel gives bitwise the single solves."""
    import paper_1801_01473_gb300 as p
    insts = []
    for k, dims in enumerate(((8, 8, 8, 8), LARGE)):
        g = p.Gauge(p.Lattice(dims), _gpu(S.gauge_links(dims, "expih", 185 + k)), "f64", 18)
        insts.append((g, None, [_gpu(S.gaussian_field(dims, 187 + k))]))
    both = p.mscg_batched(insts, [0.01, 0.5], 0.3, tol=1e-10)
    for (g, _, (b,)), (x, _) in zip(insts, both):
        one, _ = p.mscg(g, b, [0.01, 0.5], 0.3, tol=1e-10)
        assert torch.equal(x[0], one)
