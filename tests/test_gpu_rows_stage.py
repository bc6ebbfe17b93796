"""The FP64 stage of small meshes with a lane per (element, node) (csrc/rows_kernel.cuh), the default up to
a few thousand triangles, against the two-kernel stage that the oracle pins: a right-hand side and 18
SSP-RK3 steps (a replayed chunk and two steps) at sizes with one element in the last warp, a full block
and many blocks, periodic and Dirichlet with time-dependent sources, element-wise and nodal D.  Both
evaluate the same products in FP64; the tolerance is the FP64 parity tolerance, 1e-12."""
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


def _run(N, m, bc, nodal, form):
    xy, tri = unit_square_mesh(m, 0.1, 4)
    K, Np = tri.shape[0], rdg.np_of(N)
    rng = np.random.default_rng(m)
    D = rng.uniform(0.3, 1.0, (K, Np)) if nodal else np.where(rng.uniform(size=K) < 0.4, 1.0, 0.05)
    s = rdg.Solver(xy, tri, N, D, v=(0.5, -0.8), bc=bc, precision=rdg.FP64, interface=rdg.IFACE_ALG1)
    s.set_stage_form(form)
    if bc == rdg.BC_DIRICHLET:
        x, g = s.node_coords(), s.ghost_coords()
        s.set_forcing([(x[..., 0] * x[..., 1], rdg.TAU_COS, 2.0)], [(g[..., 0], rdg.TAU_SIN, 3.0), (g[..., 1], rdg.TAU_COS, 1.0)])
    u = torch.tensor(random_nodal(K, Np, 2), dtype=torch.float64, device="cuda")
    r = torch.empty_like(u)
    s.rhs_eval(u, r, 0.3)
    s.set_state(u)
    s.solve_to_time(0.1, 0.05 / m ** 2 / (N + 1) ** 4, 18)
    out = r.cpu().numpy(), s.get_state_host()
    s.synchronize()
    s.close()
    return out


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("m,bc,nodal", [(3, rdg.BC_PERIODIC, False), (4, rdg.BC_DIRICHLET, False), (9, rdg.BC_PERIODIC, True),
                                        (31, rdg.BC_DIRICHLET, False)])
def test_rows_stage_matches_two_kernels(N, m, bc, nodal):
    for a, b in zip(_run(N, m, bc, nodal, rdg.STAGE_AUTO), _run(N, m, bc, nodal, rdg.STAGE_TWO_KERNELS)):
        assert parity_err(a, b) < 1e-12
