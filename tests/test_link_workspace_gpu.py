"""Memory of the link operations (gauge force and action, smearing, chain rule): a pool of the library's own, so
that the process's default pool keeps the program's settings; given back with the last lattice; no memory
nodes in a captured FP64 gauge force or smearing, which run the per-link kernels then.

Tolerance of the captured forms against the eager ones: as for either against the oracle (products of at most 5
matrices or a chain of about 20, entries of order one to ten): 1e-12 of the largest entry.
"""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu

DIMS = (6, 10, 4, 12)
RHO, BETA = 0.15, 4.1


def _cudart():
    for name in ("libcudart.so.13", "libcudart.so", "/usr/local/cuda/lib64/libcudart.so"):
        try:
            return ctypes.CDLL(name)
        except OSError:
            continue
    pytest.skip("no shared CUDA runtime to ask")


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _setup(dt=torch.complex128):
    import paper_1801_01473_gb300 as p
    lat = p.Lattice(DIMS)
    u = torch.from_numpy(S.gauge_links(DIMS, "haar", 231)).cuda()
    rng = np.random.default_rng(232)
    grad = torch.from_numpy(rng.standard_normal(u.shape) + 1j * rng.standard_normal(u.shape)).cuda()
    return p, lat, u.to(dt), grad.to(dt)


@pytest.mark.parametrize("dt", [torch.complex128, torch.complex64])
def test_default_pool_keeps_its_threshold(dt):
    rt = _cudart()
    p, lat, u, grad = _setup(dt)
    pool, old, got = ctypes.c_void_p(), ctypes.c_uint64(), ctypes.c_uint64()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    attr = 4  # cudaMemPoolAttrReleaseThreshold
    assert rt.cudaMemPoolGetAttribute(pool, attr, ctypes.byref(old)) == 0
    assert rt.cudaMemPoolSetAttribute(pool, attr, ctypes.byref(ctypes.c_uint64(1 << 20))) == 0
    try:
        p.gauge_force(lat, u, BETA)
        levels = p.stout_smear(lat, u, RHO, 2)
        p.stout_force(lat, u, levels, RHO, grad)
        if dt == torch.complex128:
            p.gauge_action(lat, u, BETA)
        torch.cuda.synchronize()
        assert rt.cudaMemPoolGetAttribute(pool, attr, ctypes.byref(got)) == 0
        assert got.value == 1 << 20
    finally:
        rt.cudaMemPoolSetAttribute(pool, attr, ctypes.byref(old))


def test_workspace_goes_with_the_last_lattice():
    code = """
import torch
import paper_1801_01473_gb300 as p
lat = p.Lattice((16, 16, 16, 16))
u = torch.zeros((4, lat.V, 3, 3), dtype=torch.complex128, device='cuda')
u[..., 0, 0] = u[..., 1, 1] = u[..., 2, 2] = 1
out = p.gauge_force(p.Lattice((2, 2, 2, 2)), u[:, :16].contiguous(), 1.0)  # loads the kernels
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
out = p.gauge_force(lat, u, 1.0)
del out
torch.cuda.synchronize()
torch.cuda.empty_cache()
held = before - torch.cuda.mem_get_info()[0]
del lat
torch.cuda.synchronize()
left = before - torch.cuda.mem_get_info()[0]
assert held > 300 << 20, held   # 6.9 kB a site
assert left < 64 << 20, (held, left)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("op", ["force", "smear"])
def test_captured_without_memory_nodes(op):
    """The captured graph is instantiated twice (refused for a graph with memory nodes) and both run."""
    rt = _cudart()
    p, lat, u, _ = _setup()
    from paper_1801_01473_gb300.lib import lib
    want = p.gauge_force(lat, u, BETA) if op == "force" else p.stout_smear(lat, u, RHO, 2)
    out = torch.empty_like(want)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    s, graph, ex = ctypes.c_void_p(st.cuda_stream), ctypes.c_void_p(), [ctypes.c_void_p(), ctypes.c_void_p()]
    assert rt.cudaStreamBeginCapture(s, 1) == 0  # thread-local
    if op == "force":
        rc = lib().stg_gauge_force(lat.handle, 0, ctypes.c_double(BETA), _p(u), _p(out), 0, s)
    else:
        rc = lib().stg_stout_smear(lat.handle, 0, 2, ctypes.c_double(RHO), _p(u), _p(out), s)
    assert rt.cudaStreamEndCapture(s, ctypes.byref(graph)) == 0 and rc == 0
    for e in ex:
        assert rt.cudaGraphInstantiate(ctypes.byref(e), graph, ctypes.c_ulonglong(0)) == 0
        out.fill_(float("nan"))
        torch.cuda.synchronize()
        assert rt.cudaGraphLaunch(e, s) == 0
        st.synchronize()
        assert float((out - want).abs().max()) <= 1e-12 * float(want.abs().max())
    for e in ex:
        rt.cudaGraphExecDestroy(e)
    rt.cudaGraphDestroy(graph)


@pytest.mark.parametrize("dt", [torch.complex128, torch.complex64])
@pytest.mark.parametrize("kind", [0, 1])
def test_captured_action_and_chain_rule(dt, kind):
    p, lat, u, grad = _setup(dt)
    from paper_1801_01473_gb300.lib import lib
    levels = p.stout_smear(lat, u, RHO, 2)
    want = p.stout_force(lat, u, levels, RHO, grad, kind=kind)
    out = torch.empty_like(want)
    act = torch.empty(3, dtype=torch.float64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        prec = 0 if dt == torch.complex128 else 1
        rc = lib().stg_stout_force(lat.handle, prec, 2, ctypes.c_double(RHO), _p(u), _p(levels), _p(grad), _p(out), kind, s)
        rc2 = lib().stg_gauge_action(lat.handle, ctypes.c_double(BETA), _p(u), _p(act), s) if dt == torch.complex128 else 0
    assert rc == 0 and rc2 == 0
    graph.replay()
    torch.cuda.synchronize()
    tol = 1e-12 if dt == torch.complex128 else 1e-12 * 2**29
    assert float((out - want).abs().max()) <= tol * float(want.abs().max())
    if dt == torch.complex128:
        r = p.gauge_action(lat, u, BETA)
        ref = np.array([r["action"], r["plaquette_sum"], r["rectangle_sum"]])
        # sums of 6 V plaquettes and 12 V rectangles of size up to 3
        assert (np.abs(act.cpu().numpy() - ref) <= 1e-13 * 36 * lat.V).all()
