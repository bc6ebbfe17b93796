"""The launch shapes of the two-kernel FP64 stage (128-thread blocks launched programmatically at order 1
and on order-2 meshes whose blocks have an SM each, single-warp blocks otherwise), at the smallest sizes,
ragged tiles and both sides of the line (with 152 SMs 7688 and 7938 triangles at order 2): right-hand sides
and SSP-RK3 steps against the one-kernel form, the low-storage scheme against its five stages written out
on rdg_rhs_eval; both 1e-12, the same products in FP64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1912_06221_gb300 as rdg
from oracle.rhs import LSRK_A, LSRK_B
from synth import random_nodal, unit_square_mesh
from tests.test_gpu_parity import parity_err


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("N,m", [(1, 3), (1, 8), (1, 63), (2, 3), (2, 8), (2, 62), (2, 63), (3, 21)])
@pytest.mark.parametrize("nodal", [False, True])
def test_two_kernel_launches(N, m, nodal):
    xy, tri = unit_square_mesh(m, 0.1, 2)
    K, Np = tri.shape[0], rdg.np_of(N)
    rng = np.random.default_rng(m)
    D = rng.uniform(0.3, 1.0, (K, Np) if nodal else K)
    s = rdg.Solver(xy, tri, N, D, v=(0.5, -0.8), precision=rdg.FP64, interface=rdg.IFACE_ALG1)
    u = torch.tensor(random_nodal(K, Np, 2), device="cuda")
    r = torch.empty_like(u)
    dt = 0.05 / m ** 2 / (N + 1) ** 4
    out = {}
    for form in (rdg.STAGE_ONE_KERNEL, rdg.STAGE_TWO_KERNELS):
        s.set_stage_form(form)
        s.rhs_eval(u, r, 0.0)
        s.set_state(u)
        s.solve_to_time(0.0, dt, 5)
        out[form] = r.cpu().numpy(), s.get_state_host()
    for a, b in zip(out[rdg.STAGE_TWO_KERNELS], out[rdg.STAGE_ONE_KERNEL]):
        assert parity_err(a, b) < 1e-12
    s.set_integrator(rdg.LSRK54)
    s.set_state(u)
    s.solve_to_time(0.0, dt, 2)
    s.set_stage_form(rdg.STAGE_ONE_KERNEL)
    w, du = u.clone(), torch.zeros_like(u)
    for _ in range(2):
        for a, b in zip(LSRK_A, LSRK_B):
            s.rhs_eval(w, r, 0.0)
            du = a * du + dt * r
            w += b * du
    assert parity_err(s.get_state_host(), w.cpu().numpy()) < 1e-12
    s.synchronize()
    s.close()
