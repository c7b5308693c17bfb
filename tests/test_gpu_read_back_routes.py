"""lbib_get_markers into pageable and page-locked arrays of bodies below and above
the size up to which pageable ones go through the context's page-locked block:
the arrays that lbib_get_markers_async queues (the same device memory: equal
bits), each of them alone and all together.
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


def sphere(nv):
    """Octahedra (6, 18, ..., 4098 vertices) and icosahedra (10 242)."""
    if nv == 10242:
        return W.icosphere(5, 5.0, (11.7, 12.2, 12.4))
    v = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    f = [(0, 2, 4), (2, 1, 4), (1, 3, 4), (3, 0, 4), (2, 0, 5), (1, 2, 5), (3, 1, 5), (0, 3, 5)]
    while len(v) < nv:
        cache, g = {}, []

        def mid(a, b):
            key = min(a, b), max(a, b)
            if key not in cache:
                cache[key] = len(v)
                v.append(tuple((np.array(v[a]) + np.array(v[b])) / 2))
            return cache[key]

        for a, b, c in f:
            x, y, z = mid(a, b), mid(b, c), mid(c, a)
            g += [(a, x, z), (x, b, y), (z, y, c), (x, y, z)]
        f = g
    v = np.array(v, float)
    return 5.0 * v / np.linalg.norm(v, axis=1)[:, None] + np.array([11.7, 12.2, 12.4]), np.array(f, np.int32)


@pytest.mark.parametrize("locked", [(0, 0, 0), (1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("nv", [258, 4098, 10242])
def test_markers_by_either_route(lbib, nv, locked):
    v, f = sphere(nv)
    assert len(v) == nv
    ctx = lbib.Context((24, 24, 24), 0.8, bc=(0, 0, 1), wall_u=W.shear_walls(0.01))
    ctx.add_body(v, f, rigid=True, density_ratio=1.1, ref_radius=5.0)
    ctx.step(3)
    ref = [np.zeros_like(v) for _ in range(3)]
    lbib.lbib_get_markers_async(ctx.h, 0, *ref)
    ctx.sync()
    for want in ((1, 1, 1), (1, 0, 0), (0, 0, 1)):
        held = [torch.full((nv, 3), np.nan, dtype=torch.float64, pin_memory=bool(k)) for k in locked]
        out = [h.numpy() for h in held]
        lbib.lbib_get_markers(ctx.h, 0, *[a if q else None for a, q in zip(out, want)])
        for a, b, q in zip(out, ref, want):
            assert np.array_equal(a, b) if q else np.isnan(a).all()
    ctx.close()
