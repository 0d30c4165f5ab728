"""FP64 stout smearing and its chain rule by shared plaquettes (k_stout_loops, k_stout_apply,
k_stout_grad_exp, k_stout_bent, k_stout_gather) against the oracle, at the sizes where their indexing
and their choice can go wrong: extents of 2, remainders of the thread block, all extents different,
the window of volumes that stays with the per-link kernels (8^4) and both its edges; one and three
steps, and rho = 0 and its largest value, where the exponential's series is longest.

Tolerance: a smearing step is a chain of about 8 products of 3-term complex dot products on numbers
of order one (error ~1e-15 a step), the chain rule about 20 on gradients of order ten; 1e-12 of the
largest entry covers three steps with the growth of the gradient through them.
"""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import stout as ostout

pytestmark = pytest.mark.gpu


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("dims,steps,rho", [((2, 2, 2, 2), 1, 0.15), ((2, 4, 6, 8), 3, 0.15), ((6, 10, 4, 14), 2, 0.15),
                                            ((4, 4, 4, 4), 1, 0.0), ((4, 6, 4, 4), 2, 0.5), ((8, 8, 8, 8), 1, 0.15),
                                            ((8, 10, 8, 8), 1, 0.15)])
@pytest.mark.parametrize("kind", [0, 1])
def test_matches_oracle(dims, steps, rho, kind):
    import paper_1801_01473_gb300 as p
    u = S.gauge_links(dims, "haar", 161)
    rng = np.random.default_rng(162)
    grad = rng.standard_normal(u.shape) + 1j * rng.standard_normal(u.shape)
    lat = p.Lattice(dims)
    want = ostout.stout(dims, u, rho, steps)
    levels = p.stout_smear(lat, _gpu(u), rho, steps)
    for k in range(steps):
        assert np.abs(levels[k].cpu().numpy() - want[k + 1]).max() <= 1e-12
    g = ostout.stout_backward(dims, want, rho, grad)
    if kind == 0:
        z = u @ np.conj(np.swapaxes(g, -1, -2))
        g = 0.5 * (z - np.conj(np.swapaxes(z, -1, -2)))
        g = g - np.trace(g, axis1=-2, axis2=-1)[..., None, None] / 3 * np.eye(3)
    got = p.stout_force(lat, _gpu(u), levels, rho, _gpu(grad), kind=kind).cpu().numpy()
    assert np.abs(got - g).max() <= 1e-12 * np.abs(g).max()


@pytest.mark.parametrize("dims,steps", [((2, 2, 2, 2), 1), ((6, 10, 4, 14), 3), ((8, 8, 8, 10), 2)])
@pytest.mark.parametrize("kind", [0, 1])
def test_single_precision_chain_rule(dims, steps, kind):
    """The FP32 per-link kernels and their workspace fields: 2^29 times the rounding of the FP64 steps
    (~1e-15 a step and product chain), with the growth of the gradient through three steps."""
    import paper_1801_01473_gb300 as p
    u = S.gauge_links(dims, "haar", 163)
    rng = np.random.default_rng(164)
    grad = rng.standard_normal(u.shape) + 1j * rng.standard_normal(u.shape)
    lat = p.Lattice(dims)
    want = ostout.stout(dims, u, 0.15, steps)
    ug = _gpu(u).to(torch.complex64)
    levels = p.stout_smear(lat, ug, 0.15, steps)
    assert np.abs(levels[-1].cpu().numpy() - want[-1]).max() <= 5e-6
    g = ostout.stout_backward(dims, want, 0.15, grad)
    if kind == 0:
        z = u @ np.conj(np.swapaxes(g, -1, -2))
        g = 0.5 * (z - np.conj(np.swapaxes(z, -1, -2)))
        g = g - np.trace(g, axis1=-2, axis2=-1)[..., None, None] / 3 * np.eye(3)
    got = p.stout_force(lat, ug, levels, 0.15, _gpu(grad).to(torch.complex64), kind=kind).cpu().numpy()
    assert np.abs(got - g).max() <= 2e-5 * np.abs(g).max()
