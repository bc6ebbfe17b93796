"""The face form (FP32, element-wise D: one kernel per stage, csrc/face_kernels.cuh) against the FP64
per-edge kernels, which the oracle pins, at the sizes where its tiles can go wrong: less than one
128-element tile, exactly one, a ragged second one, several; a right-hand side and a solve of 19
steps (a replayed chunk of 16, then three steps that pass the records on) with both integrators;
convection, both interface rules, tensor D, Dirichlet data with time-dependent sources.  The
tolerance is the FP32 parity tolerance, 1e-5 of the largest value."""
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


def _run(N, m, prec, kind, iface, bc, integ):
    xy, tri = unit_square_mesh(m, 0.1, m)
    K = tri.shape[0]
    rng = np.random.default_rng(N)
    D = {"jump": np.where(rng.uniform(size=K) < 0.4, 1.0, 0.05), "tensor": rng.uniform(0.3, 1.0, (K, 2))}[kind]
    s = rdg.Solver(xy, tri, N, D, v=(0.6, -0.9), bc=bc, precision=prec, interface=iface)
    s.set_integrator(integ)
    if bc == rdg.BC_DIRICHLET:
        x, g = s.node_coords(), s.ghost_coords()
        s.set_forcing([(np.sin(3 * x[..., 0]) * x[..., 1], rdg.TAU_COS, 2.0), (x[..., 0], rdg.TAU_CONST, 0.0)],
                      [(g[..., 0] - g[..., 1], rdg.TAU_SIN, 3.0), (g[..., 1] ** 2, rdg.TAU_COS, 1.0)])
    u = torch.tensor(random_nodal(K, s.Np, 7).astype(np.float32), dtype=s.dtype, device="cuda")
    r = torch.empty_like(u)
    s.rhs_eval(u, r, 0.4)
    s.set_state(u)
    s.solve_to_time(0.2, 0.05 / m ** 2 / (N + 1) ** 4, 19)
    out = [r.double().cpu().numpy(), s.get_state_host().astype(np.float64)]
    s.synchronize()
    s.close()
    return out


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("m,kind,iface,bc,integ", [
    (3, "jump", rdg.IFACE_ALG1, rdg.BC_PERIODIC, rdg.SSP_RK3),
    (8, "tensor", rdg.IFACE_ALG1, rdg.BC_DIRICHLET, rdg.LSRK54),
    (9, "jump", rdg.IFACE_ALG2, rdg.BC_DIRICHLET, rdg.SSP_RK3),
    (21, "tensor", rdg.IFACE_ALG2, rdg.BC_PERIODIC, rdg.LSRK54),
    (21, "jump", rdg.IFACE_HARMONIC, rdg.BC_DIRICHLET, rdg.SSP_RK3)])
def test_face_form_matches_fp64(N, m, kind, iface, bc, integ):
    got = _run(N, m, rdg.FP32, kind, iface, bc, integ)
    want = _run(N, m, rdg.FP64, kind, iface, bc, integ)
    for a, b in zip(got, want):
        assert parity_err(a, b) < 1e-5


# one size per kernel choice beyond the tiny meshes above: more than one tile per SM, and more tiles
# than the small build holds at once (ragged last tiles)
LARGE_M = {1: 225, 2: 225, 3: 225, 4: 225, 5: 181, 6: 150}


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("large", [False, True])
@pytest.mark.parametrize("integ", [rdg.SSP_RK3, rdg.LSRK54])
def test_face_form_kernel_choice_matches_fp64(N, large, integ):
    m = LARGE_M[N] if large else 75
    got = _run(N, m, rdg.FP32, "jump", rdg.IFACE_ALG1, rdg.BC_DIRICHLET, integ)
    want = _run(N, m, rdg.FP64, "jump", rdg.IFACE_ALG1, rdg.BC_DIRICHLET, integ)
    for a, b in zip(got, want):
        assert parity_err(a, b) < 1e-5


@pytest.mark.parametrize("prec,N,integ", [(rdg.FP32, 2, rdg.SSP_RK3), (rdg.FP32, 5, rdg.LSRK54), (rdg.FP64, 3, rdg.SSP_RK3),
                                          (rdg.FP32_3XTF32, 4, rdg.SSP_RK3)])
@pytest.mark.parametrize("forced", [False, True])
def test_direct_and_replayed_solves_agree(prec, N, integ, forced):
    """The first solve of a dt launches its steps directly, the next one replays a captured chunk (16
    steps, then three more): the same kernels, so the same bits; with forcing the stage times are summed
    in another order, 1e-6 in FP32 and 1e-13 in FP64."""
    xy, tri = unit_square_mesh(11, 0.1, 3)
    s = rdg.Solver(xy, tri, N, 0.4, v=(0.3, 0.2), precision=prec)
    s.set_integrator(integ)
    if forced:
        x = s.node_coords()
        s.set_forcing([(np.sin(3 * x[..., 0]) * x[..., 1], rdg.TAU_COS, 200.0)])
    u = torch.tensor(random_nodal(s.K, s.Np, 7), dtype=s.dtype, device="cuda")
    out = []
    for _ in range(3):
        s.set_state(u)
        s.solve_to_time(0.2, 0.02 / 11 ** 2 / (N + 1) ** 4, 19)
        out.append(s.get_state_host().astype(np.float64))
    s.synchronize()
    s.close()
    assert np.array_equal(out[1], out[2])
    if forced:
        assert parity_err(out[0], out[1]) < (1e-13 if prec == rdg.FP64 else 1e-6)
    else:
        assert np.array_equal(out[0], out[1])
