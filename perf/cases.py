"""Performance cases of the framework: what its users run, through the public Python entry points.

A case is a dict of plain values:

  op      "rhs"      one right-hand side of a nodal field (the call inside a user's own integrator)
          "solve"    set the state, advance it by `steps` steps, read it back (all on the device)
          "request"  a served solve: mesh and data on the host, set up, advance, read back to the host
          "batch"    `members` independent heat problems of uneven size and order advanced together
  N       polynomial order 1..6
  m       cells per side of the unit square; every cell is two jittered triangles, K = 2 m^2
  prec    "fp32", "fp64" or "tf32" (the split 3xTF32 tensor-core form of the edge flux)
  iface   "alg1" or "alg2" (the paper's two interface rules) or "harmonic"
  D       "const" (pure heat), "circle" (jump across a circle, convection-diffusion) or "tensor"
          (element-wise diagonal tensor, convection-diffusion)
  bc      "periodic" or "dirichlet" (manufactured solution: two source terms, ghost data)
  integ   "ssp" (SSP-RK3) or "lsrk" (the paper's five-stage low-storage scheme)

exact() restates the method in 64-bit torch: reference operators, per-edge reconstruction
operators, the semi-discrete right-hand side and the integrators.
"""
import functools
import math

import numpy as np
import torch

import paper_1912_06221_gb300 as rdg

VELOCITY = (1.0, 0.5)


def listed():
    return [
        # smallest call: one right-hand side of the 512-triangle heat mesh, all launch latency
        dict(name="rhs_N2_m16", op="rhs", N=2, m=16, prec="fp32", iface="alg2", D="const", bc="periodic", integ="ssp",
             steps=0),
        # the plain FP64 heat problem: 200 steps on 512 triangles
        dict(name="heat_N2_m16_fp64", op="solve", N=2, m=16, prec="fp64", iface="alg2", D="const", bc="periodic",
             integ="ssp", steps=200),
        # low order on a medium mesh, element count no multiple of any tile
        dict(name="pulse_N1_m181", op="solve", N=1, m=181, prec="fp32", iface="alg1", D="circle", bc="periodic",
             integ="ssp", steps=50),
        # the manufactured-solution problem of the precision sweep: Dirichlet data and sources
        dict(name="manufactured_N3_m96", op="solve", N=3, m=96, prec="fp32", iface="alg2", D="const", bc="dirichlet",
             integ="ssp", steps=64),
        # the circle pulse on 131072 triangles, the headline workload, in a chunk of 100 steps
        dict(name="pulse_N4_m256", op="solve", N=4, m=256, prec="fp32", iface="alg1", D="circle", bc="periodic",
             integ="ssp", steps=100),
        # the same mesh with the edge flux on the tensor cores
        dict(name="pulse_N4_m256_tf32", op="solve", N=4, m=256, prec="tf32", iface="harmonic", D="circle",
             bc="periodic", integ="ssp", steps=32),
        # the FP64 run that FP32 results are checked against
        dict(name="pulse_N4_m128_fp64", op="solve", N=4, m=128, prec="fp64", iface="alg1", D="circle", bc="periodic",
             integ="ssp", steps=20),
        # anisotropic diffusion with the paper's integrator on a ragged mesh
        dict(name="tensor_N5_m101_lsrk", op="solve", N=5, m=101, prec="fp32", iface="alg2", D="tensor", bc="periodic",
             integ="lsrk", steps=30),
        # highest order, medium mesh
        dict(name="pulse_N6_m181", op="solve", N=6, m=181, prec="fp32", iface="alg1", D="circle", bc="periodic",
             integ="ssp", steps=40),
        # the largest served mesh, 1M triangles: a few steps of it
        dict(name="pulse_N3_m707", op="solve", N=3, m=707, prec="fp32", iface="alg1", D="circle", bc="periodic",
             integ="ssp", steps=24),
        # a served request of ordinary size: set-up, 50 steps and both copies
        dict(name="request_N4_m61", op="request", N=4, m=61, prec="fp32", iface="alg1", D="circle", bc="periodic",
             integ="ssp", steps=50),
        # uneven heat problems stepped together
        dict(name="batch_12", op="batch", N=6, m=128, members=12, mix=2, prec="fp32", iface="alg2", D="const",
             bc="periodic", integ="ssp", steps=20),
    ]


def draw(rng):
    """Another case of the same ranges: sizes spread over their logarithm, every order, type and option."""
    op = rng.choices(["solve", "rhs", "request", "batch"], [12, 3, 2, 2])[0]
    prec = rng.choices(["fp32", "fp64", "tf32"], [12, 3, 1])[0] if op == "solve" else "fp32"
    N = rng.randint(1, 5 if prec == "tf32" else 6)
    lo, hi = (16, 512) if prec == "fp32" else (16, 181)
    lo, hi = {"request": (22, 181), "batch": (24, 128)}.get(op, (lo, hi))
    m = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    while op == "solve" and 2 * m * m * (N + 1) * (N + 2) // 2 > 12_000_000:
        m = int(0.8 * m)
    D = "const" if op == "batch" else rng.choices(["circle", "const", "tensor"], [6, 3, 2 if prec != "tf32" else 0])[0]
    iface = "alg2" if op == "batch" else rng.choice(["harmonic", "alg2"]) if prec == "tf32" else "alg1"
    if D in ("const", "tensor") and prec != "tf32" and op != "batch":
        iface = rng.choice(["alg1", "alg2"])
    if D == "circle" and iface == "alg2":
        iface = "harmonic"          # Algorithm 2 is unstable across a large jump
    bc = "dirichlet" if D == "const" and op == "solve" and rng.random() < 0.5 else "periodic"
    c = dict(op=op, N=N, m=m, prec=prec, iface=iface, D=D, bc=bc, integ="ssp", steps=0)
    if op != "rhs":
        c["steps"] = int(round(math.exp(rng.uniform(math.log(8), math.log(100)))))
        cost = 3.0 * 2 * m * m * (N + 1) * (N + 2) / 2 * (20.0 if prec == "fp64" else 1.0)
        if op == "batch":
            c.update(members=rng.randint(3, 16), mix=rng.randrange(1 << 20))
            cost *= 0.5 * c["members"]
        c["steps"] = max(4, min(c["steps"], int(5.5e8 / cost)))
    if op == "solve" and prec != "tf32" and rng.random() < 0.2:
        c["integ"] = "lsrk"
        c["steps"] = max(4, c["steps"] * 3 // 5)
    return c


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------

def _mesh(m, seed):
    """Jittered m x m x 2 triangulation of the unit square: vertices [(m+1)^2, 2], triangles [2 m^2, 3]."""
    h = 1.0 / m
    jj, ii = np.meshgrid(np.arange(m + 1), np.arange(m + 1), indexing="ij")
    xy = np.stack([ii.ravel() * h, jj.ravel() * h], axis=1).astype(np.float64)
    inner = ((ii > 0) & (ii < m) & (jj > 0) & (jj < m)).ravel()
    xy[inner] += np.random.default_rng(seed).uniform(-0.1 * h, 0.1 * h, (int(inner.sum()), 2))
    cj, ci = np.meshgrid(np.arange(m), np.arange(m), indexing="ij")
    a = (cj * (m + 1) + ci).ravel()
    tri = np.empty((2 * m * m, 3), np.int32)
    tri[0::2] = np.stack([a, a + 1, a + m + 2], axis=1)
    tri[1::2] = np.stack([a, a + m + 2, a + m + 1], axis=1)
    return xy, tri


def _members(case):
    """The single problems of a case: itself, or a batch's uneven members."""
    if case["op"] != "batch":
        return [case]
    rng = np.random.default_rng(case["mix"])
    return [dict(case, op="solve", N=int(rng.integers(1, case["N"] + 1)),
                 m=int(round(math.exp(rng.uniform(math.log(8), math.log(case["m"]))))), scale=float(rng.uniform(0.2, 1.0)))
            for _ in range(case["members"])]


def _coefficients(case, xy, tri, seed):
    """(D array, v): element-wise D of the case's kind."""
    K = tri.shape[0]
    if case["D"] == "const":
        return np.full(K, case.get("scale", 1.0)), (0.0, 0.0)
    if case["D"] == "tensor":
        return np.random.default_rng(seed + 1).uniform(0.3, 1.0, (K, 2)), VELOCITY
    c = xy[tri].mean(axis=1)
    return np.where(np.hypot(c[:, 0] - 0.5, c[:, 1] - 0.5) < 0.25, 1.0, 1e-4), VELOCITY


def _dt(case):
    return 0.1 / case["m"] ** 2 / (case["N"] + 1) ** 4


def _real(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _node_coords(N, xy, tri):
    """Physical nodes [K, Np, 2] (float64, on the device) of the triangles."""
    r, s = (torch.as_tensor(a, device="cuda") for a in _nodes(N))
    p = torch.as_tensor(xy, device="cuda")[torch.as_tensor(tri, device="cuda").long()]
    lam = torch.stack([-(r + s) / 2, (r + 1) / 2, (s + 1) / 2], dim=1)
    return torch.einsum("il,kld->kid", lam, p)


def _field(case, xy, tri, seed):
    """The case's input field [K, Np]: seeded normal nodal values for a lone right-hand side, the
    manufactured solution, or a seeded sum of Gaussian pulses."""
    N, K = case["N"], tri.shape[0]
    if case["op"] == "rhs":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return torch.randn(K, (N + 1) * (N + 2) // 2, generator=gen, device="cuda", dtype=_real(case))
    X = _node_coords(N, xy, tri)
    if case["bc"] == "dirichlet":
        return _sine(X).to(_real(case)).contiguous()
    rng = np.random.default_rng(seed + 2)
    u = torch.zeros(X.shape[:2], device="cuda", dtype=torch.float64)
    for cx, cy, w, a in zip(rng.uniform(0.3, 0.7, 4), rng.uniform(0.3, 0.7, 4), rng.uniform(0.04, 0.12, 4),
                            rng.uniform(0.5, 1.5, 4)):
        u += a * torch.exp(-((X[..., 0] - cx) ** 2 + (X[..., 1] - cy) ** 2) / w ** 2)
    return u.to(_real(case)).contiguous()


def _sine(X):
    return torch.sin(math.pi * X[..., 0]) * torch.sin(math.pi * X[..., 1])


def _setup(case, xy, tri, D, v):
    """The framework's context of a case: mesh, operators, integrator, forcing."""
    s = rdg.Solver(xy, tri, case["N"], D, v=v, bc=rdg.BC_DIRICHLET if case["bc"] == "dirichlet" else rdg.BC_PERIODIC,
                   period=(1.0, 1.0), precision={"fp32": rdg.FP32, "fp64": rdg.FP64, "tf32": rdg.FP32_3XTF32}[case["prec"]],
                   interface={"alg1": rdg.IFACE_ALG1, "alg2": rdg.IFACE_ALG2, "harmonic": rdg.IFACE_HARMONIC}[case["iface"]])
    if case["integ"] == "lsrk":
        s.set_integrator(rdg.LSRK54)
    if case["bc"] == "dirichlet":
        f = _sine(_node_coords(case["N"], xy, tri)).cpu().numpy()
        g = _sine(torch.as_tensor(s.ghost_coords())).numpy()
        s.set_forcing(src=[(-f, 2, 1.0), (2 * math.pi ** 2 * f, 1, 1.0)], ghost=[(g, 1, 1.0)])
    return s


def prepare(case, seed):
    state = {"case": case, "dt": _dt(case), "solvers": [], "u": []}
    for i, c in enumerate(_members(case)):
        xy, tri = _mesh(c["m"], seed + 100 * i)
        D, v = _coefficients(c, xy, tri, seed + 100 * i)
        u = _field(c, xy, tri, seed + 100 * i)
        if case["op"] == "request":
            state.update(xy=xy, tri=tri, D=D, v=v, u_host=u.cpu().pin_memory(), out_host=torch.empty_like(u, device="cpu").pin_memory())
            return state
        state["solvers"].append(_setup(c, xy, tri, D, v))
        state["u"].append(u)
    if case["op"] == "rhs":
        state["rhs"] = state["solvers"][0].new_field()
    if case["op"] == "batch":
        state["batch"] = rdg.Batch()
        for c, s in zip(_members(case), state["solvers"]):
            state["batch"].add(s, _dt(c))
    return state


def run(state):
    case = state["case"]
    if case["op"] == "rhs":
        state["solvers"][0].rhs_eval(state["u"][0], state["rhs"], 0.0)
        return state["rhs"]
    if case["op"] == "request":
        s = _setup(case, state["xy"], state["tri"], state["D"], state["v"])
        s.set_state(state["u_host"])
        s.solve_to_time(0.0, state["dt"], case["steps"])
        s.get_state(state["out_host"])
        s.close()
        return state["out_host"]
    for s, u in zip(state["solvers"], state["u"]):
        s.set_state(u)
    if case["op"] == "batch":
        state["batch"].step(case["steps"])
    else:
        state["solvers"][0].solve_to_time(0.0, state["dt"], case["steps"])
    return [s.get_state() for s in state["solvers"]]


def work(case):
    """Bytes: the field in and out, and once each element's five metric coefficients, its Jacobian and three
    neighbours and each edge's eight geometric numbers.  Operations per right-hand side: the method's
    products with the reference matrices, Dr, Ds and the two weak derivatives (4 Np^2 multiply-adds per
    element), LIFT (3 Np Nfp) and the folded edge operator (2 Np Nfp per edge)."""
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _members(case):
        N, K = c["N"], 2 * c["m"] ** 2
        Np, Nfp, E, size = (N + 1) * (N + 2) // 2, N + 1, 1.5 * K, 8 if c["prec"] == "fp64" else 4
        evals = 1 if c["op"] == "rhs" else c["steps"] * (5 if c["integ"] == "lsrk" else 3)
        total["bytes"] += 2 * K * Np * size + K * (6 * size + 12) + E * 8 * size
        total["flops"] += 2.0 * evals * (K * (4 * Np * Np + 3 * Np * Nfp) + E * 2 * Np * Nfp)
    return total


# ---------------------------------------------------------------------------------------
# The method in 64 bits
# ---------------------------------------------------------------------------------------

def _lgl(N):
    leg = np.polynomial.legendre
    return np.array([-1.0, 1.0]) if N == 1 else np.concatenate([[-1.0], np.sort(leg.Legendre.basis(N).deriv().roots().real), [1.0]])


@functools.lru_cache(None)
def _nodes(N):
    """Warp & Blend nodes (alpha = 0) of the reference triangle, row by row."""
    i, j = np.array([(i, j) for i in range(N + 1) for j in range(N + 1 - i)]).T
    lam = np.stack([i / N, 1 - i / N - j / N, j / N])          # weights of the top, left and right vertex
    xe = np.linspace(-1, 1, N + 1)
    fit = np.polynomial.polynomial.Polynomial(np.linalg.solve(np.vander(xe, increasing=True), _lgl(N) - xe))
    xy = np.array([[0.0, 2 / math.sqrt(3)], [-1, -1 / math.sqrt(3)], [1, -1 / math.sqrt(3)]]).T @ lam
    for k, (a, b) in enumerate(((1, 2), (2, 0), (0, 1))):      # warp along the edge a -> b
        q = lam[b] - lam[a]
        inside = np.abs(q) < 1 - 1e-10
        w = np.where(inside, 4 * lam[a] * lam[b] * fit(q) / np.where(inside, 1 - q * q, 1.0), 0.0)
        xy += np.array([[math.cos(2 * math.pi * k / 3)], [math.sin(2 * math.pi * k / 3)]]) * w
    l1 = (math.sqrt(3) * xy[1] + 1) / 3
    l2 = (-3 * xy[0] - math.sqrt(3) * xy[1] + 2) / 6
    l3 = 1 - l1 - l2
    return -l2 + l3 - l1, -l2 - l3 + l1


def _legendre(N, x):
    """Orthonormal Legendre values and derivatives, two lists of N + 1 (numpy or torch)."""
    P, D = [0 * x + 1, x], [0 * x, 0 * x + 1]
    for n in range(1, N):
        P.append(((2 * n + 1) * x * P[n] - n * P[n - 1]) / (n + 1))
        D.append(D[n - 1] + (2 * n + 1) * P[n])
    c = [math.sqrt(n + 0.5) for n in range(N + 1)]
    return [a * b for a, b in zip(c, P)], [a * b for a, b in zip(c, D)]


class _Ref:
    """Reference operators of one order.  Modes: P_a(r) P_b(s), a + b <= N, made orthonormal on the triangle."""

    def __init__(self, N):
        self.N, self.Np, self.Nfp = N, (N + 1) * (N + 2) // 2, N + 1
        x, w = np.polynomial.legendre.leggauss(2 * N + 3)
        a, b = (g.ravel() for g in np.meshgrid(x, x, indexing="ij"))
        rq, sq, wq = (1 + a) * (1 - b) / 2 - 1, b, (np.outer(w, w).ravel()) * (1 - b) / 2
        self.T = np.eye(self.Np)
        B = self.modes(rq, sq)[0]
        self.T = np.linalg.inv(np.linalg.qr(np.sqrt(wq)[:, None] * B)[1])
        r, s = self.r, self.s = _nodes(N)
        V, Vr, Vs = self.modes(r, s)
        self.V, self.Vinv = V, np.linalg.inv(V)
        Dr, Ds = Vr @ self.Vinv, Vs @ self.Vinv
        Minv = V @ V.T
        M = np.linalg.inv(Minv)
        t = _lgl(N)
        lam = np.stack([-(r + s) / 2, (r + 1) / 2, (s + 1) / 2])
        self.fmask = []
        for f in range(3):                                     # face nodes from its first to its second vertex
            on = np.flatnonzero(np.abs(lam[(f + 2) % 3]) < 1e-9)
            self.fmask.append(on[np.argsort(lam[(f + 1) % 3][on])])
        V1 = np.stack(_legendre(N, t)[0], axis=1)
        E = np.zeros((self.Np, 3 * self.Nfp))
        for f in range(3):
            E[self.fmask[f], f * self.Nfp:(f + 1) * self.Nfp] = np.linalg.inv(V1 @ V1.T)
        self.LIFT, self.Dr, self.Ds = Minv @ E, Dr, Ds
        self.Wr, self.Ws = Minv @ Dr.T @ M, Minv @ Ds.T @ M
        # reconstruction on the logical square, side 2 through the point reflection
        P = self.modes(rq, sq)[0].T * wq
        A = [P @ self.square(rq, sq)[0], P @ self.square(-rq, -sq)[0]]
        pinv = np.linalg.pinv(np.vstack(A), rcond=1e-13)
        Ap = [pinv[:, :self.Np] @ self.Vinv, pinv[:, self.Np:] @ self.Vinv]    # from side values
        Phi, PR, PS = self.square(-t, t)
        self.Q = [(PR @ Ap[k], PS @ Ap[k]) for k in range(2)]                  # u~_R, u~_S on the diagonal
        self.R = [Phi @ Ap[k] for k in range(2)]                              # u~ on the diagonal
        # Algorithm 1: gradient on sub-triangle j of the projection of u~, reconstructed again
        self.Z = [[[(1, -1)[j] * self.R[j] @ Dm @ V @ A[j] @ Ap[k] for Dm in (Dr, Ds)] for k in range(2)] for j in range(2)]

    def modes(self, r, s):
        (Pr, Dr), (Ps, Ds) = _legendre(self.N, r), _legendre(self.N, s)
        ab = [(a, b) for a in range(self.N + 1) for b in range(self.N + 1 - a)]
        st = torch.stack if isinstance(r, torch.Tensor) else np.stack
        T = torch.as_tensor(self.T, device=r.device) if isinstance(r, torch.Tensor) else self.T
        return [st([X[a] * Y[b] for a, b in ab], -1) @ T for X, Y in ((Pr, Ps), (Dr, Ps), (Pr, Ds))]

    def square(self, R, S):
        (PR, DR), (PS, DS) = _legendre(self.N, R), _legendre(self.N, S)
        n = range(self.N + 1)
        return [np.stack([X[a] * Y[b] for a in n for b in n], 1) for X, Y in ((PR, PS), (DR, PS), (PR, DS))]


def _edges(m, periodic):
    """(k1, f1, k2, f2, shift): the structured mesh's edges; k2 = -1 on the Dirichlet boundary."""
    cj, ci = (g.ravel() for g in np.meshgrid(np.arange(m), np.arange(m), indexing="ij"))
    lo = 2 * (cj * m + ci)
    zero = np.zeros((m * m, 2))
    out = [(lo, 2, lo + 1, 0, zero)]                            # the cell's diagonal
    right, up = 2 * (cj * m + (ci + 1) % m), 2 * (((cj + 1) % m) * m + ci)
    sh = [zero + np.stack([ci == m - 1, 0 * ci], 1), zero + np.stack([0 * cj, cj == m - 1], 1)]
    for k1, f1, k2, f2, edge, shift in ((lo, 1, right + 1, 2, ci == m - 1, sh[0]), (lo + 1, 1, up, 0, cj == m - 1, sh[1])):
        keep = np.ones(m * m, bool) if periodic else ~edge
        out.append((k1[keep], f1, k2[keep], f2, shift[keep]))
        if not periodic:
            out.append((k1[edge], f1, np.full(edge.sum(), -1), 1, zero[edge]))
    if not periodic:
        out += [(lo[cj == 0], 0, np.full(m, -1), 1, zero[:m]), (lo[ci == 0] + 1, 2, np.full(m, -1), 1, zero[:m])]
    cat = lambda q: np.concatenate([np.broadcast_to(o[q], o[0].shape if q < 4 else o[4].shape) for o in out])  # noqa: E731
    return [torch.as_tensor(cat(q), device="cuda") for q in range(5)]


def _cross(a, b):
    return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]


def _apex(e1, e2, q1, q2r):
    """Apex of the largest parallelogram with diagonal e1 e2: highest point common to (e1, e2, q1) and (e1, e2, q2r)."""
    def inside(p, q):
        det = _cross(e2 - e1, q - e1)
        l2, l3 = _cross(p - e1, q - e1) / det, _cross(e2 - e1, p - e1) / det
        return (l2 > -1e-12) & (l3 > -1e-12) & (1 - l2 - l3 > -1e-12)

    def meet(a0, a1, b0, b1):
        det = _cross(a1 - a0, b1 - b0)
        return a0 + (_cross(b0 - a0, b1 - b0) / torch.where(det == 0, torch.full_like(det, 1e-300), det))[..., None] * (a1 - a0)

    best, high = e1.clone(), torch.zeros_like(e1[..., 0])
    for p in (q1, q2r, meet(e1, q1, e2, q2r), meet(e2, q1, e1, q2r)):
        h = torch.where(torch.isfinite(p).all(-1) & inside(p, q1) & inside(p, q2r), _cross(e2 - e1, p - e1), torch.zeros_like(high))
        best, high = torch.where((h > high)[..., None], p, best), torch.maximum(h, high)
    return best


class _Exact:
    """The semi-discrete problem of one case."""

    def __init__(self, case, xy, tri, D, v):
        ref = self.ref = _Ref(case["N"])
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=torch.float64)  # noqa: E731
        Np, Nfp = ref.Np, ref.Nfp
        self.X = t(xy)[torch.as_tensor(tri, device="cuda").long()]
        X, K = self.X, tri.shape[0]
        self.k1, self.f1, self.k2, self.f2, shift = _edges(case["m"], case["bc"] == "periodic")
        self.ghost = self.k2 < 0
        k2 = torch.where(self.ghost, self.k1, self.k2)
        D = t(D)
        D = D if D.ndim == 2 else D[:, None].expand(K, 2)
        xr, xs = (X[:, 1] - X[:, 0]) / 2, (X[:, 2] - X[:, 0]) / 2
        J = _cross(xr, xs)
        gr, gs = torch.stack([xs[:, 1], -xs[:, 0]], 1) / J[:, None], torch.stack([-xr[:, 1], xr[:, 0]], 1) / J[:, None]
        vv = t(v)
        self.coef = [c[:, None] for c in (gr @ vv, gs @ vv, (D * gr * gr).sum(1), (D * gr * gs).sum(1), (D * gs * gs).sum(1))]
        corner = lambda k, f, c: X[k, (f + c) % 3]  # noqa: E731
        e1, e2, q1 = (corner(self.k1, self.f1, c) for c in range(3))
        q2 = torch.where(self.ghost[:, None], e1 + e2 - q1, corner(k2, self.f2, 2) + shift)
        p1 = _apex(e1, e2, q1, e1 + e2 - q2)
        d = e2 - e1
        length = d.norm(dim=1)
        n = torch.stack([d[:, 1], -d[:, 0]], 1) / length[:, None]
        self.Jf, vn = length / 2, n @ vv
        xR, xS = (e1 - p1) / 2, (e2 - p1) / 2
        Jp = _cross(xR, xS)[:, None]
        gR, gS = torch.stack([xS[:, 1], -xS[:, 0]], 1) / Jp, torch.stack([-xR[:, 1], xR[:, 0]], 1) / Jp
        D1, D2 = D[self.k1], D[k2]
        E = self.k1.shape[0]
        self.W = torch.empty(E, Nfp, 2 * Np, device="cuda", dtype=torch.float64)
        lam = t(np.stack([-(ref.r + ref.s) / 2, (ref.r + 1) / 2, (ref.s + 1) / 2], 1))
        Dt = 2 * D1 * D2 / (D1 + D2) if case["iface"] == "harmonic" else (D1 + D2) / 2
        for lo in range(0, E, 32768):
            c = slice(lo, min(E, lo + 32768))
            for side in range(2):
                ea, eb, q, p, f = (e1, e2, q1, p1, self.f1) if side == 0 else (e2, e1, q2, e1 + e2 - p1, self.f2)
                ea, eb, q, p, f = ea[c], eb[c], q[c], p[c], f[c]
                det = _cross(eb - ea, q - ea)
                apex = torch.stack([torch.zeros_like(det), _cross(p - ea, q - ea) / det, _cross(eb - ea, p - ea) / det], 1)
                apex[:, 0] = 1 - apex[:, 1] - apex[:, 2]
                # weights of the sub-triangle's nodes on (ea, eb, q): node weights on (apex, ea, eb)
                w = lam[None, :, 0:1] * apex[:, None, :]
                w[..., 0] += lam[:, 1]
                w[..., 1] += lam[:, 2]
                own = torch.gather(w, 2, ((torch.arange(3, device="cuda")[None] - f[:, None]) % 3)[:, None, :].expand(-1, Np, -1))
                Vs = ref.modes(2 * own[..., 1] - 1, 2 * own[..., 2] - 1)[0] @ t(ref.Vinv)
                mat = lambda a, b: t(a)[None] * b[:, None, None]  # noqa: E731
                if case["iface"] == "alg1":
                    C = 0
                    for j, Dj in enumerate((D1[c], D2[c])):
                        C = C + mat(ref.Z[j][side][0], (n[c] * Dj * gR[c]).sum(1)) + mat(ref.Z[j][side][1], (n[c] * Dj * gS[c]).sum(1))
                else:
                    C = mat(ref.Q[side][0], (n[c] * Dt[c] * gR[c]).sum(1)) + mat(ref.Q[side][1], (n[c] * Dt[c] * gS[c]).sum(1))
                Wk = -self.Jf[c][:, None, None] * (C @ Vs)
                up = (self.Jf * vn)[c] * ((vn[c] >= 0) if side == 0 else (vn[c] < 0))
                for i in range(Nfp):
                    cols = torch.as_tensor(np.stack([m[i if side == 0 else Nfp - 1 - i] for m in ref.fmask]), device="cuda")[f]
                    Wk[torch.arange(Wk.shape[0], device="cuda"), i, cols] += up
                self.W[c, :, side * Np:(side + 1) * Np] = Wk
        self.mats = [t(a.T) for a in (ref.Dr, ref.Ds, ref.Wr, ref.Ws, ref.LIFT)]
        self.J, self.n_elem = J, K
        self.src, self.gdata = [], []
        if case["bc"] == "dirichlet":
            real = _real(case)
            f = _sine(_node_coords(case["N"], xy, tri))
            self.src = [((-f).to(real).double(), math.sin), ((2 * math.pi ** 2 * f).to(real).double(), math.cos)]
            g = torch.stack([(e1 + e2 - q1), e2, e1], 1)[self.ghost]
            self.gdata = _sine(torch.einsum("il,kld->kid", lam, g)).to(real).double()

    def rhs(self, u, time):
        Dr, Ds, Wr, Ws, LIFT = self.mats
        ar, as_, grr, grs, gss = self.coef
        ur, us = u @ Dr, u @ Ds
        out = (ar * u - grr * ur - grs * us) @ Wr + (as_ * u - grs * ur - gss * us) @ Ws
        pair = torch.cat([u[self.k1], u[self.k2.clamp(min=0)]], 1)
        if len(self.gdata):
            pair[self.ghost, self.ref.Np:] = self.gdata * math.cos(time)
        q = torch.bmm(self.W, pair[:, :, None])[:, :, 0]
        fb = torch.zeros(self.n_elem, 3, self.ref.Nfp, device="cuda", dtype=torch.float64)
        fb[self.k1, self.f1] = q
        inner = ~self.ghost
        fb[self.k2[inner], self.f2[inner]] = -q[inner].flip(1)
        out -= fb.reshape(self.n_elem, -1) @ LIFT / self.J[:, None]
        for f, tau in self.src:
            out += f * tau(time)
        return out


_CK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385, -1275806237668 / 842570457699)
_CK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498, 3134564353537 / 4481467310338,
         2277821191437 / 14882151754819)
_CK_C = (0.0, 1432997174477 / 9575080441755, 2526269341429 / 6820363962896, 2006345519317 / 3224310063776, 2802321613138 / 2924317926251)


def exact(case, seed):
    out = []
    for i, c in enumerate(_members(case)):
        xy, tri = _mesh(c["m"], seed + 100 * i)
        D, v = _coefficients(c, xy, tri, seed + 100 * i)
        p = _Exact(c, xy, tri, D, v)
        u, dt = _field(c, xy, tri, seed + 100 * i).double(), _dt(c)
        for n in range(c["steps"]):
            time = n * dt
            if c["integ"] == "lsrk":
                du = torch.zeros_like(u)
                for a, b, ct in zip(_CK_A, _CK_B, _CK_C):
                    du = a * du + dt * p.rhs(u, time + ct * dt)
                    u = u + b * du
            else:
                w = u + dt * p.rhs(u, time)
                w = 0.75 * u + 0.25 * (w + dt * p.rhs(w, time + dt))
                u = u / 3 + 2 / 3 * (w + dt * p.rhs(w, time + dt / 2))
        if c["op"] == "rhs":
            return p.rhs(u, 0.0)
        out.append(u)
    return out[0].cpu() if case["op"] == "request" else out
