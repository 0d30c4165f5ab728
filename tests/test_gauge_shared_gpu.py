"""The FP64 gauge force from staples shared between links (k_gauge_staples, k_gauge_bent,
k_gauge_gather) against the loop-by-loop oracle, at the sizes where its indexing can go wrong: the
smallest lattice, extents of 2 (both neighbours the same site), remainders of the thread block, all
extents different; links that are no SU(3) matrices, since the factors may not assume unitarity;
and a volume whose workspace takes several passes over the planes.

Tolerance: G is a sum of 24 products of at most 5 matrices, each of 3-term complex dot products, so
its rounding error is below 24 * 5 * 8 * 2^-53 ~ 1e-13 of the largest product; 1e-12 leaves the
cancellation between the plaquette and rectangle parts.
"""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import gauge as og

pytestmark = pytest.mark.gpu

BETA = 4.1


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 4), (2, 4, 6, 8), (6, 10, 4, 14)])
@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("kind", [0, 1])
def test_matches_loops(dims, general, kind):
    import paper_1801_01473_gb300 as p
    u = S.gauge_links(dims, "haar", 151)
    if general:
        rng = np.random.default_rng(152)
        u = u + 0.3 * (rng.standard_normal(u.shape) + 1j * rng.standard_normal(u.shape))
    want = og.gradient(dims, u, BETA) if kind == 1 else og.force(dims, u, BETA)
    got = p.gauge_force(p.Lattice(dims), _gpu(u), BETA, kind=kind).cpu().numpy()
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()


def test_several_passes():
    """32^4 takes the planes in two passes: the Lie-algebra force is the projection of U G^dag."""
    import paper_1801_01473_gb300 as p
    dims = (32, 32, 32, 32)
    g = torch.Generator(device="cuda").manual_seed(153)
    u = torch.view_as_complex(torch.randn((4, 32**4, 3, 3, 2), dtype=torch.float64, device="cuda", generator=g)) * 0.4
    lat = p.Lattice(dims)
    grad, force = (p.gauge_force(lat, u, BETA, kind=k) for k in (1, 0))
    # translation by one site in t commutes with the force
    step = 32**3
    moved = p.gauge_force(lat, torch.roll(u, step, dims=1), BETA, kind=1)
    assert float((torch.roll(grad, step, dims=1) - moved).abs().max()) == 0.0
    z = (u[..., :, :, None] * grad.conj().transpose(-1, -2)[..., None, :, :]).sum(-2)
    want = 0.5 * (z - z.conj().transpose(-1, -2))
    tr = torch.diagonal(want, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3
    want = want - tr * torch.eye(3, device="cuda")
    assert float((force - want).abs().max()) <= 1e-13 * float(z.abs().max())


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 10, 4, 14)])
@pytest.mark.parametrize("kind", [0, 1])
def test_single_precision_matches_loops(dims, kind):
    """The per-link kernel (FP32), whose factors are grouped too: 2^-24 in place of 2^-53 above."""
    import paper_1801_01473_gb300 as p
    u = S.gauge_links(dims, "haar", 154).astype(np.complex64)
    want = og.gradient(dims, u, BETA) if kind == 1 else og.force(dims, u, BETA)
    got = p.gauge_force(p.Lattice(dims), _gpu(u), BETA, kind=kind).cpu().numpy()
    assert np.abs(got - want).max() <= 24 * 5 * 8 * 2.0**-24 * np.abs(want).max()
