"""D launches on more blocks than one grid dimension counts (65535): 64^4 has 8388608 sites per parity,
131072 blocks of 64 sites, so small-block shapes go in several launches, the last one partial.  Unit
links, where D is a signed difference of neighbours; <p, A p> checks the partial sums' places.

Tolerance: FP32, sums of 16 terms of order one twice: 32 * 2^-24 of the largest value.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

DIMS = (64, 64, 64, 64)
MASS = 0.3


def _free_d(psi, par, out_par):
    """D of a field [Lt, Lz, Ly, Lx, 3] that lives on the other parity, at parity out_par."""
    t, z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda") for n in DIMS], indexing="ij")
    out = torch.zeros_like(psi)
    for mu, (axis, s) in enumerate(((3, 0 * x), (2, x), (1, x + y), (0, x + y + z))):
        eta = (1.0 - 2.0 * (s % 2)).to(psi.real.dtype)
        fwd, bwd = eta.clone(), eta.clone()
        if mu == 3:
            fwd[-1] *= -1
            bwd[0] *= -1
        out += 0.5 * (fwd[..., None] * torch.roll(psi, -1, axis) - bwd[..., None] * torch.roll(psi, 1, axis))
    out[par != out_par] = 0
    return out


@pytest.mark.parametrize("shape", ["64", "128", "256"])
def test_normal_operator(shape, monkeypatch):
    import paper_1801_01473_gb300 as p
    monkeypatch.setenv("STG_DSLASH_SHAPE", shape)
    v = 64**4
    lat = p.Lattice(DIMS)
    unit = torch.eye(3, dtype=torch.complex128, device="cuda").expand(4, v, 3, 3).contiguous()
    g = p.Gauge(lat, unit, "f32", 12)
    del unit
    gen = torch.Generator(device="cuda").manual_seed(201)
    psi = torch.view_as_complex(torch.randn((v // 2, 3, 2), dtype=torch.float64, device="cuda", generator=gen))
    inp = p.pack(lat, psi, "f32")
    out, tmp, pq = g.new_field(), g.new_field(), torch.empty(1, dtype=torch.float64, device="cuda")
    p.normal_op_(g, MASS, 0.0, out, inp, tmp, pq)
    grid = torch.meshgrid(*[torch.arange(n, device="cuda") for n in DIMS], indexing="ij")
    par = sum(grid) % 2
    full = torch.zeros((*DIMS, 3), dtype=torch.complex64, device="cuda")
    full[par == 0] = psi.to(torch.complex64)
    want = MASS**2 * full - _free_d(_free_d(full, par, 1), par, 0)
    want = want[par == 0]
    got = p.unpack(lat, out).to(torch.complex64)
    assert float((got - want).abs().max()) <= 32 * 2.0**-24 * float(want.abs().max())
    exact = float((psi.conj() * got.to(torch.complex128)).real.sum())
    assert abs(float(pq) - exact) <= 1e-6 * abs(exact)
