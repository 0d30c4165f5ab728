"""The FP64 gauge force and action where their workspace takes the planes in several passes of several planes
(32^4: three a pass), by value: the force against the FP32 per-link kernel, whose loops know no planes, and the
action against sums in plain torch.

Tolerance: FP32 rounding of 24 products of at most 5 matrices of 3-term complex dot products, 24 * 5 * 8 * 2^-24 of
the largest entry; the action's 6 V plaquettes and 12 V rectangles of size at most |U|^4 and |U|^6 carry
~40 * 2^-53 each.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

BETA, DIMS = 4.1, (32, 32, 32, 32)


def _links():
    g = torch.Generator(device="cuda").manual_seed(251)
    return torch.view_as_complex(torch.randn((4, 32**4, 3, 3, 2), dtype=torch.float64, device="cuda", generator=g)) * 0.4


def _up(f, mu):
    return torch.roll(f.reshape(*DIMS[::-1], *f.shape[1:]), -1, dims=3 - mu).reshape(f.shape)


@pytest.mark.parametrize("kind", [0, 1])
def test_force_by_value(kind):
    import paper_1801_01473_gb300 as p
    lat, u = p.Lattice(DIMS), _links()
    got = p.gauge_force(lat, u, BETA, kind=kind)
    want = p.gauge_force(lat, u.to(torch.complex64), BETA, kind=kind).to(torch.complex128)
    assert float((got - want).abs().max()) <= 24 * 5 * 8 * 2.0**-24 * float(want.abs().max())


def test_action_by_value():
    import paper_1801_01473_gb300 as p
    u = _links()
    got = p.gauge_action(p.Lattice(DIMS), u, BETA)
    plaq = rect = size_p = size_r = 0.0
    for mu in range(4):
        for nu in range(4):
            if nu == mu:
                continue
            corner, other = u[mu] @ _up(u[nu], mu), u[nu] @ _up(u[mu], nu)
            if mu < nu:
                plaq += float((corner * other.conj()).sum().real)
                size_p += float((corner.abs() * other.abs()).sum())
            low, high = u[mu] @ _up(corner, mu), other @ _up(_up(u[mu], nu), mu)
            rect += float((low * high.conj()).sum().real)
            size_r += float((low.abs() * high.abs()).sum())
    assert abs(got["plaquette_sum"] - plaq) <= 40 * 2.0**-53 * size_p
    assert abs(got["rectangle_sum"] - rect) <= 40 * 2.0**-53 * size_r
    want = -BETA / 3 * (2 * 5 / 6 * plaq - rect / 12)
    assert abs(got["action"] - want) <= 40 * 2.0**-53 * BETA * (size_p + size_r)
