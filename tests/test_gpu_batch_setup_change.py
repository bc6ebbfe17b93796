"""A batch whose members' set-up changes between steps: forcing replaced, integrator switched, operators
built again with another D.  The next batch step takes the new set-up (its buffers, its integrator for
replayed and direct steps alike), in the persistent and in the graph form: every member's state equals
that of the same calls on a context of its own, within the FP32 parity tolerance 1e-5 (FP64 member:
1e-12).  A member left without operators is refused."""
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


STEPS = 6            # with chunks of 4: one replay and two direct steps


class Problem:
    def __init__(self, N, m, prec):
        xy, tri = unit_square_mesh(m, 0.1, N)
        self.dt = 0.1 / m ** 2 / (N + 1) ** 4
        self.D = np.where(np.arange(tri.shape[0]) % 3 == 0, 1.0, 0.3)
        self.s = rdg.Solver(xy, tri, N, self.D, v=(0.4, 0.3), bc=rdg.BC_DIRICHLET, precision=prec, interface=rdg.IFACE_ALG1)
        self.s.set_state(random_nodal(self.s.K, self.s.Np, 5))
        self.force(1.0)

    def force(self, a):
        x, g = self.s.node_coords(), self.s.ghost_coords()
        w = 0.3 / (STEPS * self.dt)                   # a change of the state of order one, and times that matter
        self.s.set_forcing([(a * w * x[..., 0], rdg.TAU_COS, w)], [(a * g[..., 1], rdg.TAU_SIN, w), (g[..., 0], rdg.TAU_CONST, 0.0)])

    def rebuild(self):
        D = np.ascontiguousarray(2.0 * self.D[::-1])
        self.s._call("rdg_operator_setup", self.s.N, D.ctypes.data_as(rdg.rdg._P), 0.4, 0.3, self.s.precision, rdg.IFACE_HARMONIC)
        self.s.set_state(random_nodal(self.s.K, self.s.Np, 6))


CHANGES = [lambda p: None, lambda p: p[0].force(-2.0), lambda p: p[1].s.set_integrator(rdg.LSRK54),
           lambda p: (p[0].rebuild(), p[0].force(0.5)), lambda p: p[1].s.set_integrator(rdg.SSP_RK3)]


@pytest.mark.parametrize("mode", [rdg.BATCH_AUTO, rdg.BATCH_GRAPH])
@pytest.mark.parametrize("precs", [(rdg.FP32, rdg.FP32), (rdg.FP32, rdg.FP64)])
def test_batch_takes_members_changed_setup(mode, precs):
    sizes = [(2, 9), (4, 7)]
    both = [[Problem(N, m, q) for (N, m), q in zip(sizes, precs)] for _ in range(2)]
    alone, mem = both
    b = rdg.Batch(chunk=4)
    for p in mem:
        b.add(p.s, p.dt)
    b.set_mode(mode)
    last = None
    for i, change in enumerate(CHANGES):
        for p in both:
            change(p)
        b.step(STEPS)
        b.synchronize()
        now = []
        for p, q, prec in zip(alone, mem, precs):
            p.s.solve_to_time(i * STEPS * p.dt, p.dt, STEPS)
            now.append(p.s.get_state_host())
            assert parity_err(q.s.get_state_host(), now[-1]) < (1e-12 if prec == rdg.FP64 else 1e-5), (i, prec)
        if last is not None:                              # the steps do change the states
            assert all(parity_err(x, y) > 1e-2 for x, y in zip(now, last))
        last = now
    mem[0].s._call("rdg_mesh_upload", 3, np.array([0.0, 0, 1, 0, 0, 1]).ctypes.data_as(rdg.rdg._P), 1,
                   np.array([0, 1, 2], np.int32).ctypes.data_as(rdg.rdg._P), rdg.BC_DIRICHLET, None)
    with pytest.raises(rdg.RdgError) as e:
        b.step(1)
    assert e.value.code == rdg.rdg.RDG_ESTATE
    b.close()
    for p in alone + mem:
        p.s.close()
