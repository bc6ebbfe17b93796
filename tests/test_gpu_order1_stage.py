"""FP32 order 1: a stage on its own (rdg_rk_stage, part 1 of a split stage) is one launch that evaluates the
neighbours' parts itself; inside a step the parts come from records.  The same arithmetic: stages one by one
equal whole steps bit by bit, at less than a tile, a tile's edge, ragged tiles and many blocks, with a jump
of D (Algorithm 1) or a tensor, periodic and with time-dependent sources and Dirichlet data; a right-hand
side agrees with FP64 to the FP32 parity tolerance 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1912_06221_gb300 as rdg
from synth import random_nodal, unit_square_mesh
from tests.test_gpu_parity import parity_err


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("m", [3, 4, 8, 21, 150])
@pytest.mark.parametrize("tensor", [False, True])
@pytest.mark.parametrize("bc", [rdg.BC_PERIODIC, rdg.BC_DIRICHLET])
def test_lone_stage_equals_step(m, tensor, bc):
    xy, tri = unit_square_mesh(m, 0.1, m)
    K = tri.shape[0]
    rng = np.random.default_rng(1)
    D = rng.uniform(0.3, 1.0, (K, 2)) if tensor else np.where(rng.uniform(size=K) < 0.4, 1.0, 0.05)
    s = {}
    for p in (rdg.FP32, rdg.FP64):
        s[p] = rdg.Solver(xy, tri, 1, D, v=(0.6, -0.9), bc=bc, precision=p, interface=rdg.IFACE_ALG1)
        if bc == rdg.BC_DIRICHLET:
            x, g = s[p].node_coords(), s[p].ghost_coords()
            s[p].set_forcing([(x[..., 0], rdg.TAU_COS, 2.0)], [(g[..., 0] - g[..., 1], rdg.TAU_SIN, 3.0), (g[..., 1], rdg.TAU_CONST, 0.0)])
    u = random_nodal(K, 3, 7).astype(np.float32)
    rhs = []
    for q in s.values():
        v = torch.tensor(u, dtype=q.dtype, device="cuda")
        r = torch.empty_like(v)
        q.rhs_eval(v, r, 0.4)
        rhs.append(r.double().cpu().numpy())
    assert parity_err(*rhs) < 1e-5
    a, dt, out = s[rdg.FP32], 0.003 / m ** 2, []
    for how in ("step", "stage", "part"):
        a.set_state(u)
        for n in range(3):
            t = 0.1 + n * dt
            if how == "step":
                a.rk_step(t, dt)
            for st in range(3 if how != "step" else 0):
                if how == "stage":
                    a.rk_stage(st, t, dt)
                else:
                    a.rk_stage_part(st, 0, t, dt)
                    a.rk_stage_part(st, 1, t, dt)
        out.append(a.get_state_host())
    for q in s.values():
        q.synchronize()
        q.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
