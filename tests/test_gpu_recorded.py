"""Recorded trajectories (lbib_step_markers) of rigid bodies, of bodies with
centroid markers and of the second body of a context, over calls that start
in and out of the six-step graph's phase, with arrays left out, against a
context read after every step.  The two contexts differ only in the order of
the atomic spreading sums, so the tolerances are those of the recorded capsule
in the parity tests.
"""
import numpy as np
import pytest

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


def context(lbib, kind):
    ctx = lbib.Context((30, 28, 33), 0.8, bc=(0, 0, 1), wall_u=W.shear_walls(0.01), precision=lbib.LBIB_FP64)
    v, f = W.icosphere(2, 4.0, (14.6, 13.4, 15.8))
    if kind == "two":
        ctx.add_body(*W.icosphere(1, 3.0, (6.2, 21.3, 16.1)), rigid=True, ref_radius=3.0)
    rigid = kind != "centroid"
    if rigid:
        ctx.add_body(v, f, rigid=True, ref_radius=4.0, density_ratio=1.3, gravity=(0.0, 0.0, -1e-5))
    else:
        ctx.add_body(v, f, rigid=False, ref_radius=4.0, ks0=1e-4, Eb=0.01, kv=1.0, density_ratio=1.0, centroid_markers=1, mass_model=1)
    return ctx, len(ctx.nv) - 1


@pytest.mark.parametrize("kind", ["rigid", "centroid", "two"])
def test_recorded_against_reads(lbib, kind):
    calls = [14, 4, 13, 1]
    ref, b = context(lbib, kind)
    want = []
    for _ in range(sum(calls)):
        ref.step(1)
        want.append(ref.markers(b))
    ref.close()
    ctx, b = context(lbib, kind)
    nv, done = ctx.nv[b], 0
    for j, n in enumerate(calls):
        got = [np.full((n, nv, 3), np.nan) for _ in range(3)]
        skip = j % 3  # one array left out in each call but the first
        lbib.lbib_step_markers(ctx.h, n, b, *[None if q == skip and j else a for q, a in enumerate(got)])
        ctx.sync()
        for k in range(n):
            for q, (a, w) in enumerate(zip(got, want[done + k])):
                if q == skip and j:
                    assert np.isnan(a).all()
                elif q == 0:
                    assert np.abs(a[k] - w).max() < 1e-13 * np.abs(w).max()
                else:
                    assert np.abs(a[k] - w).max() < 1e-10 * max(np.abs(w).max(), 1e-3)
        done += n
    ctx.close()
