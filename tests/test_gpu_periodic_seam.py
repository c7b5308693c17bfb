"""The IB force at the node before a periodic boundary where the axis has
n % 8 == 1 nodes: that node alone is the last tile of the axis, and a marker
nearest to it has support in three tiles along the axis.  A small cube
whose leading face is nearest to that node and whose other markers are far
enough behind not to flag the tile.  (Larger cubes, of 12 triangles as well,
carry so much area a marker that the run diverges.)  Against the oracle,
tolerances of the other parity tests (FP64 1e-12 of the flow's scale, FP32
1e-5).
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


@pytest.mark.parametrize("how", ["alone", "batch", "persistent"])
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("axes,centroid", [((0,), 0), ((1,), 0), ((0, 1), 0), ((0, 1, 2), 0), ((0,), 1)])
def test_force_in_the_last_tile_is_applied(lbib, axes, centroid, prec, how):
    n = tuple(17 if a in axes else 22 for a in range(3))
    side, lead = (3.6, 15.65) if centroid else (2.4, 16.05)
    c = np.array([lead - side / 2 if a in axes else 11.27 for a in range(3)])
    v, f = W.cube_mesh(side)
    z, y, x = np.meshgrid(*[np.arange(m) for m in n[::-1]], indexing="ij")
    u = np.zeros(z.shape + (3,))
    for a, (p, q, s) in enumerate(((y, z, 0), (z, x, 1), (x, y, 2))):
        u[..., a] = 4e-3 * (np.sin(2 * np.pi * p / n[(a + 1) % 3]) + np.cos(2 * np.pi * q / n[(a + 2) % 3])) + 2e-3
    body = W.Body(v + c, f, rigid=True, density_ratio=1.2, ref_radius=3.0, centroid_markers=centroid)
    case = W.Case("seam", n, 0.8, (0, 0, 0), np.zeros((6, 3)), precision=prec, bodies=[body], u0=u.reshape(-1, 3))
    steps = 13 if how == "persistent" else 5  # the persistent kernel takes six at a time
    ctx = lbib.Context.from_case(case)
    if how == "alone":
        ctx.step(steps)
    else:
        b = lbib.Batch([ctx])
        if how == "persistent":
            b.set_persistent(1)
        b.step(steps)
        b.sync()
        b.close()
    s = oracle.Sim(case.n, case.tau, gext=case.gext, bc=case.bc, wall_u=case.wall_u.ravel())
    s.set_fields(*case.initial_fields())
    s.add_body(body.verts, f, **body.kwargs())
    assert s.step(steps) == 0
    (Xg, Vg, Fg), (Xo, Vo, Fo) = ctx.markers(0), s.markers(0)
    ug, uo = ctx.fields()[1], s.fields()[1]
    ctx.close()
    s.close()
    xtol, utol = (1e-12 * 17, 1e-12 * 1e-2) if prec == W.PREC_FP64 else (1e-4, 1e-5 * 1e-2)
    assert np.abs(Xg - Xo).max() < xtol
    for a, b in ((Vg, Vo), (Fg, Fo), (ug, uo)):
        assert np.abs(a - b).max() < utol
