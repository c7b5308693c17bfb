"""Sweeps of small FP64 lattices against the FP64 oracle at the sizes where
the launch changes: single rows, consecutive nodes in blocks of one warp, and
blocks of 128 nodes, with rows a node short of and past a warp, whole warps,
and a last block that is not full.  Every launch sums a node's populations in
the same order, so the tolerance is that of the other parity tests (1e-12
relative).
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


@pytest.mark.parametrize("bc", [(0, 1, 0), (1, 1, 1)])
@pytest.mark.parametrize("n", [(24, 24, 24), (31, 30, 30), (33, 30, 28), (32, 32, 32), (63, 25, 12), (25, 24, 28),
                               (45, 33, 30), (44, 60, 40), (5, 41, 3)])
def test_small_fp64_sweeps(lbib, n, bc):
    rng = np.random.default_rng(sum(n))
    wall_u = 0.02 * rng.standard_normal((6, 3))
    for f in range(6):
        wall_u[f, f // 2] = 0.0  # tangential wall motion
    case = W.case_empty(n=n, tau=0.9, bc=bc, wall_u=wall_u, seed=4, amplitude=5e-3)
    ctx = lbib.Context.from_case(case, precision=lbib.LBIB_FP64)
    ctx.step(9)
    fg, (rg, ug) = ctx.populations(), ctx.fields()
    ctx.close()
    s = oracle.Sim(case.n, case.tau, gext=case.gext, bc=case.bc, wall_u=case.wall_u.ravel())
    s.set_fields(*case.initial_fields())
    assert s.step(9) == 0
    fo, (ro, uo) = s.populations(), s.fields()
    s.close()
    assert np.abs(fg - fo).max() < 1e-12 * np.abs(fo).max()
    assert np.abs(rg - ro).max() < 1e-12 * np.abs(ro).max()
    assert np.abs(ug - uo).max() < 1e-12 * max(np.abs(uo).max(), 1e-2)
