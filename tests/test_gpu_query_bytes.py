"""rdg_query_bytes against the device memory a context takes from the stream-ordered pool: an upper bound
for every order, precision, boundary and forcing, as set up by default, with a per-edge stage form set
before the set-up, and twice it with the form changed afterwards.  The pool hands out multiples of 512
bytes; 20 allocations and the fixed words of a context are well within 16 KiB."""
import ctypes
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1912_06221_gb300 as rdg
from synth import unit_square_mesh

SLACK = 16 << 10


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def pool_used():
    """Bytes in use in device 0's default memory pool (CU_MEMPOOL_ATTR_USED_MEM_CURRENT = 7)."""
    gc.collect()                      # contexts of other tests
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    pool, used = ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolGetAttribute(pool, 7, ctypes.byref(used)) == 0
    return used.value


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("prec,iface", [(rdg.FP32, rdg.IFACE_ALG1), (rdg.FP64, rdg.IFACE_ALG2), (rdg.FP32_3XTF32, rdg.IFACE_ALG2),
                                        (rdg.FP32_3XTF32, rdg.IFACE_ALG1)])
@pytest.mark.parametrize("bc", [rdg.BC_PERIODIC, rdg.BC_DIRICHLET])
def test_query_bytes_bounds_what_a_context_takes(N, prec, iface, bc):
    xy, tri = unit_square_mesh(100, 0.1, 1)
    torch.cuda.current_stream()
    before = pool_used()
    s = rdg.Solver(xy, tri, N, 0.5, precision=prec, interface=iface, bc=bc)
    nsrc, nghost = 0, 0
    if bc == rdg.BC_DIRICHLET:
        nsrc, nghost = 2, 3
        s.set_forcing([(np.zeros((s.K, s.Np)), rdg.TAU_COS, 1.0)] * nsrc, [(np.zeros((s.B, s.Np)), rdg.TAU_COS, 1.0)] * nghost)
    bound = rdg.query_bytes(N, s.K, s.E, s.B, prec, nsrc, nghost)
    taken = pool_used() - before
    assert 0 < taken <= bound + SLACK
    s.set_stage_form(rdg.STAGE_TWO_KERNELS)
    assert pool_used() - before <= 2 * bound + SLACK
    D = np.full(s.K, 0.5)
    s._call("rdg_operator_setup", N, D.ctypes.data_as(ctypes.c_void_p), 0.0, 0.0, prec, iface)
    if nsrc:
        s.set_forcing([(np.zeros((s.K, s.Np)), rdg.TAU_COS, 1.0)] * nsrc, [(np.zeros((s.B, s.Np)), rdg.TAU_COS, 1.0)] * nghost)
    assert pool_used() - before <= bound + SLACK
    s.set_stage_form(rdg.STAGE_AUTO)
    u = torch.zeros((s.K, s.Np), dtype=s.dtype, device="cuda")
    s.set_state(u)
    s.solve_to_time(0.0, 1e-7, 2)                       # the form that was not set up runs
    s.synchronize()
    assert not s.get_state_host().any()
    s.close()
    assert pool_used() == before
