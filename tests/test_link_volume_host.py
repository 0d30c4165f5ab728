"""The link operations number sites in 32 bits: a lattice of 2^31 sites, which stg_lattice_create allows, is refused
before anything is launched (no GPU needed)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def L():
    from paper_1801_01473_gb300 import build as b
    b.build()
    from paper_1801_01473_gb300.lib import lib
    return lib()


def test_refused(L):
    from paper_1801_01473_gb300.lib import STG_ERR_SHAPE, STG_F32, STG_F64
    lat = ctypes.c_void_p()
    assert L.stg_lattice_create((ctypes.c_int32 * 4)(256, 256, 256, 128), 1, ctypes.byref(lat)) == 0
    a, b, c = (ctypes.c_void_p(k << 20) for k in (1, 2, 3))  # never read
    rcs = [L.stg_gauge_action(lat, 5.6, a, b, None)]
    for prec in (STG_F64, STG_F32):
        rcs += [L.stg_gauge_force(lat, prec, 5.6, a, b, 0, None), L.stg_stout_smear(lat, prec, 1, 0.1, a, b, None),
                L.stg_stout_force(lat, prec, 1, 0.1, a, a, b, c, 0, None)]
    L.stg_lattice_destroy(lat)
    assert set(rcs) == {STG_ERR_SHAPE}
