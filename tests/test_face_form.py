"""The face form's element-local arithmetic (csrc/face_ops.h on the operators that csrc/gen_face.cpp
writes), compiled for the host, against the FP64 oracle's right-hand side: every order, interface
rule and kind of element-wise D, with convection.

FP64: the same real-number operator up to rounding, 1e-11 of the largest value (the oracle's pins
hold to 1e-12; the operators' constants are composed in another order).  FP32: 1e-5, the parity
tolerance of the FP32 kernels.  A constant state without convection gives exactly zero."""
import ctypes
import shutil
import subprocess
import os

import numpy as np
import pytest

from oracle.mesh import Mesh
from oracle.rhs import Problem
from synth import random_nodal, unit_square_mesh

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "..", "paper_1912_06221_gb300", "csrc")
CXX = shutil.which("g++")


def _run(cmd, **kw):
    r = subprocess.run(cmd, capture_output=True, text=True, **kw)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout


@pytest.fixture(scope="module")
def gen(tmp_path_factory):
    d = tmp_path_factory.mktemp("face")
    _run([CXX, "-std=c++17", "-O1", os.path.join(SRC, "gen_face.cpp"), os.path.join(SRC, "refops.cpp"), "-o", str(d / "gen")])
    return d


def _lib(gen, N):
    so = gen / ("f%d.so" % N)
    if not so.exists():
        (gen / ("ops%d.h" % N)).write_text(_run([str(gen / "gen"), str(N)]))
        _run([CXX, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", SRC, "-DORDER=%d" % N,
              '-DFACE_OPS="%s"' % (gen / ("ops%d.h" % N)), os.path.join(HERE, "face_host.cpp"), "-o", str(so)])
    return ctypes.CDLL(str(so))


def _parameters(pr, iface):
    """Face parameters, neighbours and element coefficients from the oracle's geometry."""
    me, eo = pr.mesh, pr.eops
    K = me.K
    D = pr.D if pr.D.ndim == 2 else np.repeat(pr.D[:, None], 2, axis=1)
    par, nbr = np.zeros((K, 3, 7)), np.zeros((K, 3), np.int64)
    for e, (k1, f1, k2, f2, _, _) in enumerate(me.edges):
        n, (Rx, Ry, Sx, Sy) = eo.n1[e], eo.Rx[e]
        Jf = 0.5 * np.hypot(*(eo.e2[e] - eo.e1[e]))
        D1, D2 = D[k1], D[k2]
        if iface == "alg2":
            D1 = D2 = 0.5 * (D1 + D2)
        elif iface == "harmonic":
            D1 = D2 = 2 * D1 * D2 / (D1 + D2)
        oR, oS, nR, nS = (-Jf * (n[0] * d[0] * gx + n[1] * d[1] * gy) for d in (D1, D2) for gx, gy in ((Rx, Ry), (Sx, Sy)))
        if iface == "alg1":
            A, B, C, Dd = (oR + oS + nR + nS) / 4, (oR - oS + nR - nS) / 4, (oR + oS - nR - nS) / 4, (oR - oS - nR + nS) / 4
        else:
            A, B, C, Dd = (oR + oS) / 2, (oR - oS) / 2, 0.0, 0.0
        s = Jf * (n @ pr.v)
        for k, f, kn, fn, (al, be), sg in ((k1, f1, k2, f2, eo.ab1[e], 1), (k2, f2, k1, f1, eo.ab2[e], -1)):
            par[k, f] = (be - al) / 2, -(al + be) / 2, A, B, sg * C, sg * Dd, sg * s
            nbr[k, f] = 4 * kn + fn
    X = me.V
    xr, xs = (X[:, 1] - X[:, 0]) / 2, (X[:, 2] - X[:, 0]) / 2
    J = xr[:, 0] * xs[:, 1] - xr[:, 1] * xs[:, 0]
    gr, gs = np.stack([xs[:, 1], -xs[:, 0]], 1) / J[:, None], np.stack([-xr[:, 1], xr[:, 0]], 1) / J[:, None]
    geo = np.stack([gr @ pr.v, gs @ pr.v, (D * gr * gr).sum(1), (D * gr * gs).sum(1), (D * gs * gs).sum(1), 1 / J], 1)
    return par, nbr, np.ascontiguousarray(geo)


@pytest.mark.skipif(CXX is None, reason="no host compiler")
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("kind,iface", [("const", "alg2"), ("jump", "alg1"), ("jump", "harmonic"), ("tensor", "alg1"),
                                        ("tensor", "alg2")])
def test_face_form_matches_oracle(gen, N, kind, iface):
    xy, tri = unit_square_mesh(4, 0.1, 5)
    K, Np = tri.shape[0], (N + 1) * (N + 2) // 2
    rng = np.random.default_rng(N)
    D = {"const": np.full(K, 0.7), "jump": np.where(rng.uniform(size=K) < 0.4, 1.0, 1e-3),
         "tensor": rng.uniform(0.2, 1.0, (K, 2))}[kind]
    pr = Problem(Mesh(xy, tri, N), D, v=(0.8, -0.5), interface=iface)
    par, nbr, geo = _parameters(pr, iface)
    lib = _lib(gen, N)
    u = random_nodal(K, Np, 3).astype(np.float32).astype(np.float64)
    want = pr.rhs(u, 0.0)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731

    def call(v, dt, par):
        v = np.ascontiguousarray(v, dt)
        out, rec = np.zeros_like(v), np.zeros((K, 3, N + 2), dt)
        (lib.rhs64 if dt == np.float64 else lib.rhs32)(int(iface == "alg1"), ctypes.c_int64(K), p(v), p(par), p(nbr), p(geo),
                                                       p(out), p(rec))
        return out

    for dt, tol in ((np.float64, 1e-11), (np.float32, 1e-5)):
        got = call(u, dt, par).astype(np.float64)
        assert np.abs(got - want).max() < tol * np.abs(want).max()
    still = par.copy()
    still[..., 6] = 0.0
    geo[:, :2] = 0.0
    assert not call(np.full((K, Np), 0.37), np.float32, still).any()
