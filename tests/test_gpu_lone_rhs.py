"""A lone right-hand side between the two parts of a split stage (rdg_rk_stage_part): the stage's
pending intermediate data is not the call's to overwrite.  FP32 split meshes above the sizes where
every lone right-hand side is one launch, rdg_rhs_eval_static and rdg_rhs_eval, SSP-RK3 and the
low-storage scheme: the state after a step with the calls in between has the same bits as without
them, and the calls' results the same bits as calls made on their own."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1912_06221_gb300 as rdg
from paper_1912_06221_gb300.partition import SplitSolver, build_plan, face_adjacency, rcb_partition
from synth import random_nodal, unit_square_mesh


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("N,m", [(1, 150), (3, 150), (4, 110), (6, 75)])
@pytest.mark.parametrize("entry", ["rdg_rhs_eval_static", "rdg_rhs_eval"])
@pytest.mark.parametrize("integ", [rdg.SSP_RK3, rdg.LSRK54])
def test_lone_rhs_between_stage_parts(N, m, entry, integ):
    xy, tri = unit_square_mesh(m, 0.1, 3)
    K = tri.shape[0]
    D = np.where(np.arange(K) % 3 == 0, 1.0, 0.2)
    plan = build_plan(rcb_partition(xy, tri, 2), face_adjacency(xy, tri), 0, 2)
    sp = SplitSolver(xy, tri, N, D, plan, v=(0.5, -0.3), precision=rdg.FP32)
    s = sp.s
    s.set_integrator(integ)
    u0 = random_nodal(K, s.Np, 2)
    w = torch.tensor(random_nodal(s.K, s.Np, 9), dtype=torch.float32, device="cuda")
    dt = 0.02 / m ** 2 / (N + 1) ** 4
    call = getattr(s.lib, entry)

    def rhs():
        r = torch.full_like(w, float("nan"))
        assert call(s.ctx, ctypes.c_void_p(w.data_ptr()), ctypes.c_void_p(r.data_ptr()), 0.0) == 0
        return r

    def step(between):
        sp.set_owned_state(u0)
        got = []
        for st in range(3 if integ == rdg.SSP_RK3 else 5):
            s.rk_stage_part(st, 0, 0.0, dt)
            if between:
                got.append(rhs())
            s.rk_stage_part(st, 1, 0.0, dt)
        return sp.owned_state(), got

    alone = rhs()
    plain, _ = step(False)
    mixed, got = step(True)
    s.synchronize()
    assert np.array_equal(plain, mixed)
    assert all(torch.equal(g, alone) for g in got)
    s.close()


@pytest.mark.parametrize("N,m", [(3, 150), (5, 75)])
@pytest.mark.parametrize("steps_before", [1, 2])
def test_replayed_rhs_between_stage_parts(N, m, steps_before):
    """The same with a right-hand side that was captured earlier, before a solve of an even or odd number
    of stages."""
    xy, tri = unit_square_mesh(m, 0.1, 3)
    plan = build_plan(rcb_partition(xy, tri, 2), face_adjacency(xy, tri), 0, 2)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        sp = SplitSolver(xy, tri, N, np.full(len(tri), 0.4), plan, v=(0.5, -0.3), precision=rdg.FP32, stream=st)
        s = sp.s
        w = torch.tensor(random_nodal(s.K, s.Np, 9), dtype=torch.float32, device="cuda")
        r = torch.empty_like(w)
        s.rhs_eval(w, r, 0.0)
        st.synchronize()
        alone = r.clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            s.rhs_eval(w, r, 0.0)
    dt = 0.02 / m ** 2 / (N + 1) ** 4

    def step(between):
        sp.set_owned_state(random_nodal(len(tri), s.Np, 2))
        s.solve_to_time(0.0, dt, steps_before)
        for stage in range(3):
            s.rk_stage_part(stage, 0, 0.0, dt)
            if between:
                with torch.cuda.stream(st):
                    r.zero_()
                    graph.replay()
            s.rk_stage_part(stage, 1, 0.0, dt)
        return sp.owned_state()

    plain, mixed = step(False), [step(True) for _ in range(2)]
    s.synchronize()
    assert all(np.array_equal(plain, x) for x in mixed)
    assert torch.equal(r, alone)
    s.close()
