"""The FP64 operator keeps FP64's relative accuracy in every real component, whatever the size of the links
and of the vector's components: links far below one, single small and zero links, links that do not mix
colours beside a colour far below the others, real links beside a far smaller imaginary part, sizes spread
over many decades.  Both kernels of the fixed-point form and the lattices below it.

Tolerance: a component is a sum of 48 products, each hop a chain of 6 roundings and 8 additions of the
hops, so an FP64 sum lies within 14 * 2^-53 of sum |u||v| over the products of that component.  The oracle
and the library each have that much: 32 * 2^-53.
"""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu

SMALL, LARGE = (8, 6, 8, 6), (24, 24, 24, 14)  # four threads per site; one (96768 sites per parity)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _abs_sums(dims, u, psi, out_par):
    """sum |u||v| / 2 of the products in the real and in the imaginary part of every output component."""
    v = int(np.prod(dims))
    par = np.stack(np.unravel_index(np.arange(v), dims[::-1])).sum(0) % 2
    full = np.zeros((v, 3), np.complex128)
    full[par != out_par] = psi
    grid = full.reshape(*dims[::-1], 3)
    at = par == out_par
    re, im = np.zeros((at.sum(), 3)), np.zeros((at.sum(), 3))
    for mu in range(4):
        axis = 3 - mu
        dag = np.conj(np.swapaxes(u[mu], -1, -2)).reshape(*dims[::-1], 3, 3)
        hops = ((u[mu], np.roll(grid, -1, axis)), (np.roll(dag, 1, axis).reshape(v, 3, 3), np.roll(grid, 1, axis)))
        for m, w in hops:
            m, w = m[at], w.reshape(v, 3)[at][:, :, None]
            mr, mi, wr, wi = np.abs(m.real), np.abs(m.imag), np.abs(w.real), np.abs(w.imag)
            re += 0.5 * (mr @ wr + mi @ wi)[..., 0]
            im += 0.5 * (mr @ wi + mi @ wr)[..., 0]
    return re, im


def _check(dims, u, psi):
    import paper_1801_01473_gb300 as p
    g = p.Gauge(p.Lattice(dims), _gpu(u), "f64", 18)
    for par, ref in ((1, oracle.dslash_oe), (0, oracle.dslash_eo)):
        d = p.dslash(g, par, _gpu(psi)).cpu().numpy() - ref(dims, u, psi)
        re, im = _abs_sums(dims, u, psi, par)
        assert (np.abs(d.real) <= 32 * 2.0**-53 * re).all() and (np.abs(d.imag) <= 32 * 2.0**-53 * im).all()


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), SMALL, LARGE])
@pytest.mark.parametrize("scale", [1.0, 1e-1, 1e-3, 1e-10, 1e-17, 1.7, 1e6])
def test_links_of_any_size(dims, scale):
    _check(dims, scale * S.gauge_links(dims, "haar", 191), S.gaussian_field(dims, 192))


@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("kind", ["haar", "expih"])
def test_single_small_and_zero_links(dims, kind):
    u = S.gauge_links(dims, kind, 193).copy()
    rng = np.random.default_rng(194)
    u *= np.where(rng.random(u.shape[:2]) < 0.02, 10.0 ** rng.uniform(-20, 0, u.shape[:2]), 1.0)[..., None, None]
    _check(dims, u, S.gaussian_field(dims, 195))
    u = S.gauge_links(dims, kind, 193).copy()
    u[3, -int(np.prod(dims[:3])):] = 0.0  # cut in time
    u[rng.random(u.shape[:2]) < 0.3] = 0.0
    _check(dims, u, S.gaussian_field(dims, 195))


@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("small", [0.0, 1e-3, 1e-10, 1e-20])
def test_links_that_do_not_mix(dims, small):
    """Unit links beside a small colour, a small imaginary part, and both."""
    u = S.gauge_links(dims, "unit", 0)
    psi = S.gaussian_field(dims, 196)
    for colour, part in ((True, False), (False, True), (True, True)):
        q = psi.copy()
        if colour:
            q[:, 1] *= small
        if part:
            q = q.real + 1j * small * q.imag
        _check(dims, u, q)


@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("kind", ["haar", "expih", "unit"])
def test_sizes_over_many_decades(dims, kind):
    rng = np.random.default_rng(197)
    u, psi = S.gauge_links(dims, kind, 198), S.gaussian_field(dims, 199)
    _check(dims, u, psi * 10.0 ** rng.uniform(-12, 0, psi.shape[:1])[:, None])
    _check(dims, u, psi * 10.0 ** rng.uniform(-12, 0, psi.shape))
    point = np.zeros_like(psi)
    point[3, 1] = 1.0
    _check(dims, u, point)


@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("part", [1.0, 1j, (1 + 1j) / 2])
def test_largest_sums(dims, part):
    """The largest links that have a fixed-point form (rows and columns of 2.49) and vectors of the largest numbers
    below a power of two with random signs, so that at many sites all 48 products add up: nothing overflows."""
    rng = np.random.default_rng(200)
    u = np.full((4, int(np.prod(dims)), 3, 3), 2.49 / 3 * part, np.complex128)
    u[:, 0] = S.gauge_links((2, 2, 2, 2), "haar", 200)[:, 0]  # the unit is the first link's
    sign = rng.choice([-1.0, 1.0], size=(2, int(np.prod(dims)) // 2))
    psi = (np.nextafter(2.0, 0.0) * (sign[0] + 1j * sign[1]))[:, None] * np.ones(3)
    _check(dims, u, psi)
