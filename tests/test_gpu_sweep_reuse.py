"""FP32 sweeps that run alternate steps from the lattice's end, with and
without streamed loads, by rows and by consecutive nodes, against the FP64
oracle at the sizes where the rule changes; an odd number of steps, walls
whose faces differ at both ends.  The tolerances are those of the FP32 parity
tests: 1e-5 relative on the velocity, 1e-6 on the density (a rounding of the
stored deviation is 1e-8 of it).
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


@pytest.mark.parametrize("n,bc", [((75, 73, 82), (0, 1, 1)), ((77, 73, 81), (0, 1, 1)), ((96, 77, 65), (1, 1, 1)),
                                  ((131, 129, 143), (0, 0, 1)), ((160, 96, 157), (1, 0, 1))])
def test_alternating_sweeps(lbib, n, bc):
    rng = np.random.default_rng(sum(n))
    wall_u = 0.02 * rng.standard_normal((6, 3))
    for f in range(6):
        wall_u[f, f // 2] = 0.0  # tangential wall motion
    case = W.case_empty(n=n, tau=0.9, bc=bc, wall_u=wall_u, seed=5, amplitude=5e-3)
    ctx = lbib.Context.from_case(case, precision=lbib.LBIB_FP32)
    ctx.step(5)
    rg, ug = ctx.fields()
    ctx.close()
    s = oracle.Sim(case.n, case.tau, gext=case.gext, bc=case.bc, wall_u=case.wall_u.ravel())
    s.set_fields(*case.initial_fields())
    assert s.step(5) == 0
    ro, uo = s.fields()
    s.close()
    assert np.abs(rg - ro).max() < 1e-6 * np.abs(ro).max()
    assert np.abs(ug - uo).max() < 1e-5 * np.abs(uo).max()
