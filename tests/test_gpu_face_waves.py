"""The face form on meshes with more tiles than its kernels hold at once, where a warp takes a second tile
into the same rows of shared memory: just above one wave of the large build (orders 1..4; it asks for 7
blocks of 128 elements per SM), above two waves, where the small build loops, and at orders 5, 6 (4 blocks)
above one wave of it.  Ragged last tiles, a jump of D, Dirichlet data with time-dependent sources; a
right-hand side and three steps of both integrators against the FP64 per-edge kernels, which the oracle
pins, to the FP32 parity tolerance 1e-5."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1912_06221_gb300 as rdg
from synth import unit_square_mesh, random_nodal
from tests.test_gpu_parity import parity_err


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _run(N, m, prec):
    xy, tri = unit_square_mesh(m, 0.1, m)
    K = tri.shape[0]
    D = np.where(np.random.default_rng(N).uniform(size=K) < 0.4, 1.0, 0.05)
    s = rdg.Solver(xy, tri, N, D, v=(0.6, -0.9), bc=rdg.BC_DIRICHLET, precision=prec, interface=rdg.IFACE_ALG1)
    x, g = s.node_coords(), s.ghost_coords()
    s.set_forcing([(np.sin(3 * x[..., 0]) * x[..., 1], rdg.TAU_COS, 2.0)], [(g[..., 0] - g[..., 1], rdg.TAU_SIN, 3.0)])
    u = torch.tensor(random_nodal(K, s.Np, 7).astype(np.float32), dtype=s.dtype, device="cuda")
    r = torch.empty_like(u)
    s.rhs_eval(u, r, 0.4)
    out = [r.double().cpu().numpy()]
    for integ in (rdg.SSP_RK3, rdg.LSRK54):
        s.set_integrator(integ)
        s.set_state(u)
        s.solve_to_time(0.2, 0.05 / m ** 2 / (N + 1) ** 4, 3)
        out.append(s.get_state_host().astype(np.float64))
    s.synchronize()
    s.close()
    return out


@pytest.mark.parametrize("N,waves", [(1, 1), (1, 2), (2, 1), (2, 2), (3, 1), (3, 2), (4, 1), (4, 2), (5, 1), (6, 1)])
def test_more_tiles_than_resident(N, waves):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    resident = sms * (7 if N <= 4 else 4) * 128                       # elements of one wave
    m = math.isqrt(waves * resident // 2) + 1
    m += m % 8 == 0                                                   # 2 m^2 no multiple of 128
    assert 2 * m * m > waves * resident
    for got, want in zip(_run(N, m, rdg.FP32), _run(N, m, rdg.FP64)):
        assert parity_err(got, want) < 1e-5
