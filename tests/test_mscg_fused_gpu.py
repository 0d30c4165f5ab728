"""The multi-shift solver's fused iteration kernels (up to 400 partial sums per system) on both sides
of their limit: 12800 sites per parity (400 partials) and 15360 (480), pure FP64 and mixed solves, one
system and three of unequal size, the smallest lattice; every shift's residual against the oracle.

Tolerance: the solver's own certificate is the residual of x at tol; the oracle's FP64 residual of
the same x differs by its rounding, ~1e-15 of cond * |x| at most here, far below tol = 1e-9.
"""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu

MASS, SHIFTS, TOL = 0.2, [1e-3, 0.05, 0.7], 1e-9


def _gauges(p, dims, inner, seed):
    u = S.gauge_links(dims, "expih", seed)
    lat = p.Lattice(dims)
    ut = torch.from_numpy(u).cuda()
    return u, p.Gauge(lat, ut, "f64", 18), p.Gauge(lat, ut, inner, 12) if inner else None


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (16, 16, 10, 10), (16, 16, 10, 12)])
@pytest.mark.parametrize("inner", [None, "f32"])
def test_both_sides_of_the_limit(dims, inner):
    import paper_1801_01473_gb300 as p
    u, g, gi = _gauges(p, dims, inner, 191)
    b = S.gaussian_field(dims, 192)
    x, st = p.mscg(g, torch.from_numpy(b).cuda(), SHIFTS, MASS, tol=TOL, g_inner=gi)
    assert max(st["true_resid"]) <= TOL
    for i, sg in enumerate(SHIFTS):
        assert oracle.true_residual(dims, u, MASS, sg, b, x[i].cpu().numpy()) <= 1.01 * TOL


@pytest.mark.parametrize("inner", [None, "f32"])
def test_systems_of_unequal_size(inner):
    import paper_1801_01473_gb300 as p
    insts, refs = [], []
    for k, (dims, nrhs) in enumerate((((4, 4, 6, 4), 2), ((8, 8, 8, 8), 1))):
        u, g, gi = _gauges(p, dims, inner, 193 + k)
        bs = [S.gaussian_field(dims, 195 + 2 * k + r) for r in range(nrhs)]
        insts.append((g, gi, [torch.from_numpy(b).cuda() for b in bs]))
        refs.append((dims, u, bs))
    for (x, _), (dims, u, bs) in zip(p.mscg_batched(insts, SHIFTS, MASS, tol=TOL), refs):
        for r, b in enumerate(bs):
            for i, sg in enumerate(SHIFTS):
                assert oracle.true_residual(dims, u, MASS, sg, b, x[r][i].cpu().numpy()) <= 1.01 * TOL
