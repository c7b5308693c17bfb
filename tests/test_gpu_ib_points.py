"""MLS points against the FP64 oracle where the kernels' index arithmetic and
support cut-off can go wrong: point counts around a warp and a block, bodies
across a periodic boundary, and markers with support nodes exactly at the
cut-off r_k = 1; in both kernels, four lanes a point (a context alone) and a
thread a point (a batch).  And the read-back of markers, through the
page-locked block and, for a body too large for it, by copies.

The tolerances are those of the other parity tests: FP64 1e-12 relative
(velocities against the flow's scale, at least 1e-2), FP32 1e-5 on
velocities and 1e-4 lattice units on positions.
"""
import numpy as np
import pytest

import oracle
from paper_2207_06029_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lbib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_06029_gb300 import build, lbib as L
    build.build()
    L.load()
    return L


def meshes():
    # 8 vertices and 12 triangles (32 points: one warp), 12 and 20 (52: part
    # of a block), 42 and 80 (202: a last block of ten), 162 and 320 (802)
    out = {"cube": W.cube_mesh(4.0)}
    for level in range(3):
        out["ico%d" % level] = W.icosphere(level, 3.0)
    return out


# offsets of the body's centre from the middle of the lattice: general,
# across the periodic x and y boundaries, far outside the first period, and
# with the cube's vertices (half-width 2) 0.3 from a node plane, which puts
# nodes 1.3 away, at r_k = 1, along every axis
PLACES = {"inside": (0.13, -0.27, 0.41), "across": (9.6, -10.2, 0.37), "outside": (55.3, -81.7, 0.2),
          "cutoff": (0.3, 0.3, 0.3)}


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("centroid", [0, 1])
@pytest.mark.parametrize("place", sorted(PLACES))
@pytest.mark.parametrize("mesh", ["cube", "ico0", "ico1", "ico2"])
def test_points_match_oracle(lbib, mesh, place, centroid, prec, batched):
    n = (20, 19, 22)
    v, f = meshes()[mesh]
    v = v + (np.array([10.0, 9.0, 11.0]) + np.array(PLACES[place]))[None, :]
    U = 0.01
    # a shear flow with an x-y variation, so that no sum of the fits vanishes
    z, y, x = np.meshgrid(*[np.arange(m) for m in n[::-1]], indexing="ij")
    u = np.zeros(z.shape + (3,))
    u[..., 0] = U * (2 * z / (n[2] - 1) - 1)
    win = np.sin(np.pi * z / (n[2] - 1))
    u[..., 1] = 2e-3 * win * np.sin(2 * np.pi * x / n[0])
    u[..., 2] = 2e-3 * win * np.cos(2 * np.pi * y / n[1])
    rho = 1 + 1e-3 * win * np.sin(2 * np.pi * (x / n[0] + y / n[1]))
    body = W.Body(v, f, rigid=True, density_ratio=1.2, ref_radius=3.0, centroid_markers=centroid)
    case = W.Case("points", n, 0.8, (0, 0, 1), W.shear_walls(U), precision=prec, bodies=[body],
                  rho0=rho.ravel(), u0=u.reshape(-1, 3))
    steps = 3
    ctx = lbib.Context.from_case(case)
    if batched:
        b = lbib.Batch([ctx])
        b.step(steps)
        b.sync()
        b.close()
    else:
        ctx.step(steps)
    s = oracle.Sim(case.n, case.tau, gext=case.gext, bc=case.bc, wall_u=case.wall_u.ravel())
    s.set_fields(*case.initial_fields())
    s.add_body(v, f, **body.kwargs())
    assert s.step(steps) == 0
    (Xg, Vg, Fg), (Xo, Vo, Fo) = ctx.markers(0), s.markers(0)
    ug, uo = ctx.fields()[1], s.fields()[1]
    bg, bo = ctx.body(0), s.body(0)
    ctx.close()
    s.close()
    if prec == W.PREC_FP64:
        assert np.abs(Xg - Xo).max() < 1e-12 * np.abs(Xo).max()
        tol = 1e-12 * 1e-2
    else:
        assert np.abs(Xg - Xo).max() < 1e-4
        tol = 1e-5 * 1e-2
    for a, b in ((Vg, Vo), (Fg, Fo), (ug, uo), (bg["u"], bo["u"])):
        assert np.abs(np.asarray(a) - np.asarray(b)).max() < tol


@pytest.mark.parametrize("level", [2, 6])  # 162 and 40 962 vertices: the block holds 14 500
def test_read_back_by_block_and_by_copies(lbib, level):
    """lbib_get_markers and lbib_get_body give the arrays that
    lbib_get_markers_async queues (the same device memory: equal bits), and
    the volume and area of those positions."""
    v, f = W.icosphere(level, 6.0, (12.2, 11.7, 12.4))
    ctx = lbib.Context((24, 24, 24), 0.8, bc=(0, 0, 1), wall_u=W.shear_walls(0.01))
    ctx.add_body(v, f, rigid=True, density_ratio=1.1, ref_radius=6.0)
    ctx.step(3)
    X, V, F = ctx.markers(0)
    ref = [np.zeros_like(v) for _ in range(3)]
    lbib.lbib_get_markers_async(ctx.h, 0, *ref)
    ctx.sync()
    for a, b in zip((X, V, F), ref):
        assert np.array_equal(a, b)
    only = np.zeros_like(v)
    lbib.lbib_get_markers(ctx.h, 0, None, only, None)
    assert np.array_equal(only, V)
    st = ctx.body(0)
    a, b, c = (X[f[:, k]] for k in range(3))
    assert abs(st["volume"] - np.einsum("ij,ij->i", a, np.cross(b, c)).sum() / 6) < 1e-9 * st["volume"]
    assert abs(st["area"] - 0.5 * np.linalg.norm(np.cross(b - a, c - a), axis=1).sum()) < 1e-9 * st["area"]
    ctx.close()
