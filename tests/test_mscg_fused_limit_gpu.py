"""The multi-shift solver's fused iteration kernels on both sides of their limit (6000 reads: blocks of 256 sites x
partials of 32 sites, over the systems of a launch), where phase 1, phase 2, both or neither run fused; every
shift's residual against the oracle.  Tolerance as the solver's certificate, the residual of x at tol."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S

pytestmark = pytest.mark.gpu

MASS, TOL = 0.2, 1e-9


# reads of phase 1 and (mixed) of phase 2 with n shifts: 8^4 8 * 64 = 512, 512 n; 10x12x10x12 29 * 225 = 6525;
# 10x10x12x10 24 * 188 = 4512, 4512 n
@pytest.mark.parametrize("dims,n", [((8, 8, 8, 8), 11), ((8, 8, 8, 8), 12), ((10, 10, 12, 10), 1), ((10, 12, 10, 12), 1)])
@pytest.mark.parametrize("inner", [None, "f32", "f16"])
def test_both_sides_of_the_limit(dims, n, inner):
    import paper_1801_01473_gb300 as p
    u = S.gauge_links(dims, "expih", 241)
    ut, lat = torch.from_numpy(u).cuda(), p.Lattice(dims)
    b = S.gaussian_field(dims, 242)
    shifts = list(np.logspace(-3, 0.5, n))
    x, st = p.mscg(p.Gauge(lat, ut, "f64", 18), torch.from_numpy(b).cuda(), shifts, MASS, tol=TOL,
                   g_inner=p.Gauge(lat, ut, inner, 12) if inner else None)
    assert max(st["true_resid"]) <= TOL
    for i, sg in enumerate(shifts):
        assert oracle.true_residual(dims, u, MASS, sg, b, x[i].cpu().numpy()) <= 1.01 * TOL
