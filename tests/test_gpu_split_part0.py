"""FP64 split meshes: part 0 of a stage (rdg_rk_stage_part) takes the work that needs no halo rows on all but
the small meshes where the whole stage after the exchange is shorter than what two kernels leave for it.
Overwriting an owned element's row of the stage input after part 0 leaves its neighbours' results as they
were, their fluxes being formed already; parts 0 then 1 equal the whole stage bit by bit."""
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


@pytest.mark.parametrize("N,m", [(1, 110), (2, 75), (4, 70), (5, 60), (6, 60)])
def test_part_0_takes_the_halo_free_fluxes(N, m):
    xy, tri = unit_square_mesh(m, 0.1, 4)
    plan = build_plan(rcb_partition(xy, tri, 2), face_adjacency(xy, tri), 0, 2)
    sp = SplitSolver(xy, tri, N, np.full(len(tri), 0.7), plan, v=(0.5, -0.3), precision=rdg.FP64)
    s = sp.s
    nbr = face_adjacency(xy, tri[plan.elements], rdg.BC_DIRICHLET)
    own = np.arange(s.K) < s.n_owned
    inner = own & (nbr >= 0).all(1) & own[np.maximum(nbr, 0)].all(1)            # no halo neighbour
    deep = np.flatnonzero(inner & inner[np.maximum(nbr, 0)].all(1))
    k = int(deep[deep.size // 2])
    u0 = random_nodal(len(tri), s.Np, 3)
    dt = 0.02 / m ** 2 / (N + 1) ** 4
    idx = torch.tensor([k], dtype=torch.int32, device="cuda")
    other = torch.full((1, s.Np), 5.0, dtype=torch.float64, device="cuda")
    rows = torch.tensor(nbr[k], dtype=torch.int32, device="cuda")
    every = torch.arange(s.n_owned, dtype=torch.int32, device="cuda")

    def stage(how):
        sp.set_owned_state(u0)
        if how == "whole":
            s.rk_stage(0, 0.0, dt)
        else:
            s.rk_stage_part(0, 0, 0.0, dt)
            if how == "overwritten":
                s.rows_scatter(other.data_ptr(), idx, 1, s.stage_buffer(0))
            s.rk_stage_part(0, 1, 0.0, dt)
        out = []
        for ix in (rows, every):
            o = torch.empty((ix.numel(), s.Np), dtype=torch.float64, device="cuda")
            s.rows_gather(s.stage_buffer(1), ix, ix.numel(), o.data_ptr())
            out.append(o)
        s.synchronize()
        return out

    parts, over, whole = stage("parts"), stage("overwritten"), stage("whole")
    assert torch.equal(parts[1], whole[1])
    assert torch.equal(parts[0], over[0])
    s.close()
