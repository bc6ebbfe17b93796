"""The same solve twice on one context: the first of a dt launches its steps directly, the second replays
captured chunks of 16 steps.  Same bits, with time-dependent sources and Dirichlet data too, in every
precision and both integrators, with whole chunks only, with remaining steps, and from a start time at
which the stage times round (0.1 has an error of 1e-17, times frequencies up to 1e6: the steps taken one by
one agree to 1e-10 in FP64)."""
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


@pytest.mark.parametrize("prec,N,kind", [(rdg.FP32, 1, "elem"), (rdg.FP32, 3, "elem"), (rdg.FP32, 6, "elem"), (rdg.FP32, 2, "nodal"),
                                         (rdg.FP32, 4, "tensor"), (rdg.FP64, 3, "tensor"), (rdg.FP64, 2, "elem"), (rdg.FP64, 4, "nodal"), (rdg.FP32_3XTF32, 3, "elem")])
@pytest.mark.parametrize("integ", [rdg.SSP_RK3, rdg.LSRK54])
@pytest.mark.parametrize("steps", [16, 53])
def test_forced_solve_repeats_bitwise(prec, N, kind, integ, steps):
    m = 10
    xy, tri = unit_square_mesh(m, 0.1, 3)
    K = tri.shape[0]
    rng = np.random.default_rng(4)
    D = rng.uniform(0.3, 1.0, {"nodal": (K, rdg.np_of(N)), "tensor": (K, 2), "elem": K}[kind])
    s = rdg.Solver(xy, tri, N, D, v=(0.3, 0.2), bc=rdg.BC_DIRICHLET, precision=prec)
    s.set_integrator(integ)
    dt = 0.05 / m ** 2 / (N + 1) ** 4
    w = 0.37 / dt                                       # the factors change over every step
    x, g = s.node_coords(), s.ghost_coords()
    s.set_forcing([(w * np.sin(3 * x[..., 0]) * x[..., 1], rdg.TAU_COS, w), (w * x[..., 0], rdg.TAU_SIN, 0.7 * w)],
                  [(g[..., 0] - g[..., 1], rdg.TAU_SIN, w), (g[..., 1] ** 2, rdg.TAU_COS, 1.3 * w)])
    u = torch.tensor(random_nodal(K, s.Np, 7), dtype=s.dtype, device="cuda")
    out = []
    for _ in range(3):
        s.set_state(u)
        s.solve_to_time(0.1, dt, steps)
        out.append(s.get_state_host())
    s.set_state(u)
    for n in range(steps):                              # and the steps one by one, to rounding
        s.rk_step(0.1 + n * dt, dt)
    one = s.get_state_host()
    s.synchronize()
    s.close()
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[1], out[2])
    assert parity_err(one, out[0]) < (1e-10 if prec == rdg.FP64 else 1e-5)
