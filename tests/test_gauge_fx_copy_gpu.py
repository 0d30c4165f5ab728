"""The fixed-point copy of an F64 gauge of 2048 sites or more belongs to the gauge like its links: operators
neither make it nor wait for it, updates carry it along (also captured ones), and every FP64 operator on
the gauge uses it.  All comparisons are bitwise, where the calls promise the same operation."""
import ctypes

import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu

DIMS = (8, 6, 8, 6)  # 2304 sites


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _links(seed, dims=DIMS):
    return _gpu(S.gauge_links(dims, "haar", seed))


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def test_captured_update_is_seen_by_later_operators():
    """An update captured before the gauge's first operator and replayed after it."""
    import paper_1801_01473_gb300 as p
    from paper_1801_01473_gb300.lib import lib
    lat = p.Lattice(DIMS)
    buf, new = _links(201), _links(202)
    g = p.Gauge(lat, buf, "f64", 18)
    psi = _gpu(S.gaussian_field(DIMS, 203))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        assert lib().stg_gauge_update(g.handle, _p(buf), None, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    p.dslash(g, 1, psi)
    buf.copy_(new)
    graph.replay()
    fresh = p.Gauge(lat, new, "f64", 18)
    for par in (0, 1):
        assert torch.equal(p.dslash(g, par, psi), p.dslash(fresh, par, psi))


def test_captured_operator_is_the_eager_one():
    import paper_1801_01473_gb300 as p
    lat = p.Lattice(DIMS)
    g = p.Gauge(lat, _links(204), "f64", 18)
    x = p.pack(lat, _gpu(S.gaussian_field(DIMS, 205)), "f64")
    out = torch.empty_like(x)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.dslash_oe_(g, out, x)
    graph.replay()
    assert torch.equal(out, p.dslash_oe_(g, torch.empty_like(x), x))


def test_first_operator_neither_allocates_nor_waits():
    import paper_1801_01473_gb300 as p
    lat = p.Lattice(DIMS)
    x = p.pack(lat, _gpu(S.gaussian_field(DIMS, 206)), "f64")
    out, tmp = torch.empty_like(x), torch.empty_like(x)
    warm = p.Gauge(lat, _links(207), "f64", 18)
    p.normal_op_(warm, 0.1, 0.0, out, x, tmp)  # settles the launch shape
    g = p.Gauge(lat, _links(208), "f64", 18)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    torch.cuda._sleep(400_000_000)  # ~0.2 s of work ahead of the operator
    p.normal_op_(g, 0.1, 0.0, out, x, tmp)
    assert not torch.cuda.current_stream().query()  # the call returned before the work ahead of it was done
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free


@pytest.mark.parametrize("others", [[(4, 4, 6, 4)], [(24, 24, 24, 14), (4, 4, 6, 4)]])
def test_batch_with_lattices_without_a_copy(others):
    """A batched FP64 solve over lattices with and without a copy gives bitwise the single solves."""
    import paper_1801_01473_gb300 as p
    insts = []
    for k, dims in enumerate([DIMS] + others):
        u = _gpu(S.gauge_links(dims, "expih", 211 + k))
        bs = [_gpu(S.gaussian_field(dims, 215 + k + 3 * j)) for j in range(2)]
        insts.append((p.Gauge(p.Lattice(dims), u, "f64", 18), None, bs))
    both = p.mscg_batched(insts, [0.01, 0.5], 0.3, tol=1e-10)
    for (g, _, bs), (x, _) in zip(insts, both):
        for b, xb in zip(bs, x):
            one, _ = p.mscg(g, b, [0.01, 0.5], 0.3, tol=1e-10)
            assert torch.equal(xb, one)


@pytest.mark.parametrize("dims", [DIMS, (24, 24, 24, 14)])
def test_noalloc_operator_is_the_normal_operator(dims):
    import paper_1801_01473_gb300 as p
    lat = p.Lattice(dims)
    g = p.Gauge(lat, _links(221, dims), "f64", 18)
    x = p.pack(lat, _gpu(S.gaussian_field(dims, 222)), "f64")
    want, got, tmp = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    pq = torch.empty(2, dtype=torch.float64, device="cuda")
    p.normal_op_(g, 0.1, 0.03, want, x, tmp, pq[:1])
    p.normal_op_noalloc_(g, 0.1, 0.03, got, x, pq[1:])
    assert torch.equal(got, want) and float(pq[0]) == float(pq[1])
