"""Bodies with so many MLS points that the blocks' partial sums (enclosed volume,
force and moment) are added up by a launch of their own: 512 blocks of 32 to
256 points by kernel and precision.  A membrane and a rigid sphere of 10 242
(51 202 points) and 40 962 vertices (204 802), alone, batched and in the
persistent kernel, against the oracle: tolerances of the other parity tests
(FP64 1e-12, FP32 1e-5 of the flow and 1e-4 lattice units).
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


def many(level, rigid, prec):
    n = (30, 28, 32)
    v, f = W.icosphere(level, 8.0, (14.63, 13.41, 15.87))
    U = 0.01
    if rigid:
        body = W.Body(v, f, rigid=True, density_ratio=1.2, ref_radius=8.0, gravity=(0.0, 0.0, -1e-5))
    else:
        # nearly force-free springs: at this mesh density any stiffness is
        # beyond the explicit update; the volume term is what the sum feeds
        body = W.Body(v, f, ks0=1e-7, Eb=0.0, kv=0.05, ref_radius=8.0, density_ratio=1.0, mass_model=1)
    return W.Case("many", n, 0.8, (0, 0, 1), W.shear_walls(U), precision=prec, bodies=[body],
                  u0=W.couette_profile(n, U))


@pytest.fixture(scope="module")
def expected():
    memo = {}

    def get(level, rigid, steps):
        key = level, rigid, steps
        if key not in memo:
            case = many(level, rigid, W.PREC_FP64)
            s = oracle.Sim(case.n, case.tau, gext=case.gext, bc=case.bc, wall_u=case.wall_u.ravel())
            s.set_fields(*case.initial_fields())
            b = case.bodies[0]
            s.add_body(b.verts, b.tris, **b.kwargs())
            assert s.step(steps) == 0
            memo[key] = s.markers(0), s.fields()[1]
            s.close()
        return memo[key]

    return get


# how, level: k_body_sums (alone), kb_body_sums (above 65 536 points), the
# persistent kernel's items (above 131 072)
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_FP32])
@pytest.mark.parametrize("rigid", [False, True])
@pytest.mark.parametrize("how,level,steps", [("alone", 5, 3), ("alone", 6, 3), ("batch", 6, 3), ("persistent", 6, 8)])
def test_sums_over_many_points(lbib, expected, how, level, steps, rigid, prec):
    (Xo, Vo, Fo), uo = expected(level, rigid, steps)
    ctx = lbib.Context.from_case(many(level, rigid, prec))
    if how == "alone":
        ctx.step(steps)
    else:
        b = lbib.Batch([ctx])
        if how == "persistent":
            b.set_persistent(1)
        b.step(steps)
        b.sync()
        b.close()
    (X, V, F), u = ctx.markers(0), ctx.fields()[1]
    ctx.close()
    xtol, utol = (1e-12 * np.abs(Xo).max(), 1e-12 * 1e-2) if prec == W.PREC_FP64 else (1e-4, 1e-5 * 1e-2)
    assert np.abs(X - Xo).max() < xtol
    assert np.abs(V - Vo).max() < utol and np.abs(F - Fo).max() < utol
    assert np.abs(u - uo).max() < utol
