"""Checkpoints of contexts that have recorded a trajectory: the staging buffer is
scratch, so the checkpoint has the size of one taken before, loads into a
context that never recorded, and into the same context after the buffer has
grown; and a context goes on after it as the saved one does (up to the order
of the atomic spreading sums: 1e-13 relative, FP64, few steps).
"""
import struct

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


def context(lbib):
    ctx = lbib.Context((22, 20, 24), 0.8, bc=(0, 0, 1), wall_u=W.shear_walls(0.01), precision=lbib.LBIB_FP64)
    v, f = W.icosphere(2, 4.0, (10.6, 9.4, 11.8))
    ctx.add_body(v, f, rigid=True, ref_radius=4.0, density_ratio=1.3, gravity=(0.0, 0.0, -1e-5))
    return ctx


def record(lbib, ctx, n):
    out = np.empty((n, ctx.nv[0], 3))
    lbib.lbib_step_markers(ctx.h, n, 0, out)
    ctx.sync()
    return out


def close_to(a, b):
    return np.abs(a - b).max() < 1e-13 * np.abs(b).max()


def test_a_recorded_context_saves_and_loads(lbib):
    a = context(lbib)
    a.step(2)
    before = len(lbib.lbib_save(a.h))
    record(lbib, a, 9)
    saved = lbib.lbib_save(a.h)
    assert len(saved) == before
    fresh = context(lbib)
    lbib.lbib_load(fresh.h, saved)
    want = record(lbib, a, 15)  # the buffer grows
    f, X = a.populations(), a.markers(0)[0]
    assert close_to(record(lbib, fresh, 15), want)
    assert close_to(fresh.populations(), f)
    assert len(lbib.lbib_save(a.h)) == before
    lbib.lbib_load(a.h, saved)
    a.step(15)
    assert close_to(a.populations(), f) and close_to(a.markers(0)[0], X)
    a.close()
    fresh.close()


def test_bodies_added_after_a_recording_are_saved(lbib):
    """Growing the staging buffer frees the old one; an array that takes its
    address belongs to the checkpoint."""
    v, f = W.icosphere(2, 3.0, (10.6, 9.4, 11.8))

    def second(ctx):
        ctx.add_body(v + np.array([0.0, 0.0, 6.2]) * 0.9, f, rigid=True, ref_radius=3.0)

    a, b = context(lbib), context(lbib)
    a.step(2)
    b.step(2)
    record(lbib, a, 1)
    record(lbib, a, 30)
    b.step(31)
    second(a)
    second(b)
    assert len(lbib.lbib_save(a.h)) == len(lbib.lbib_save(b.h))
    saved = lbib.lbib_save(a.h)
    a.step(7)
    c = context(lbib)
    second(c)
    lbib.lbib_load(c.h, saved)
    c.step(7)
    assert close_to(c.populations(), a.populations())
    for k in range(2):
        assert close_to(c.markers(k)[0], a.markers(k)[0])
    for ctx in (a, b, c):
        ctx.close()


def test_checkpoints_that_hold_the_staging_buffer_load_as_before(lbib):
    """Older checkpoints of a recorded context end with its staging buffer;
    they load into a context with one of the same size and no other."""
    a = context(lbib)
    record(lbib, a, 5)
    saved = lbib.lbib_save(a.h)
    size = 3 * 5 * 3 * a.nv[0] * 8
    old = bytearray(saved + struct.pack("<Q", size) + bytes(size))
    count = struct.unpack_from("<i", old, 36)[0]  # the header's number of arrays
    struct.pack_into("<i", old, 36, count + 1)
    a.step(7)
    f = a.populations()
    lbib.lbib_load(a.h, bytes(old))
    a.step(7)
    assert close_to(a.populations(), f)
    fresh = context(lbib)
    for n in (0, 6):  # no staging buffer, one of another size
        if n:
            record(lbib, fresh, n)
        with pytest.raises(lbib.LbibError):
            lbib.lbib_load(fresh.h, bytes(old))
    lbib.lbib_load(fresh.h, saved)
    a.close()
    fresh.close()
