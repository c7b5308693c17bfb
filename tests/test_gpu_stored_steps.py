"""Steps that store the fields, replayed from captured graphs once their phase of
the buffer rotation stores for the third time, against steps enqueued kernel
by kernel: the fluid alone bit for bit, fields and populations; with a body up
to the order of the atomic spreading sums (1e-13 relative, FP64, 28 steps or
fewer).
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


def context(lbib, body, prec):
    n = (22, 20, 25)
    ctx = lbib.Context(n, 0.8, bc=(0, 0, 1), wall_u=W.shear_walls(0.01), precision=prec)
    ctx.set_fields(np.ones(n[0] * n[1] * n[2]) + 1e-3 * np.random.default_rng(4).uniform(-1, 1, n[0] * n[1] * n[2]),
                   W.couette_profile(n, 0.01))
    if body:
        v, f = W.icosphere(2, 4.0, (10.63, 9.41, 11.87))
        ctx.add_body(v, f, rigid=True, ref_radius=4.0, density_ratio=1.3, gravity=(0.0, 0.0, -1e-5))
    return ctx


# calls and lbib_set_output: a store at the end of each call of six (one
# phase), of four (three phases), of mixed lengths; and every third step
CALLS = [([6, 6, 6, 6], 0), ([4] * 7, 0), ([1, 5, 7, 5, 1, 6], 0), ([9, 9, 9], 3), ([2] * 13, 1)]


@pytest.mark.parametrize("calls,every", CALLS)
@pytest.mark.parametrize("body,prec", [(False, W.PREC_FP64), (False, W.PREC_FP32), (True, W.PREC_FP64)])
def test_replayed_storing_steps(lbib, body, prec, calls, every):
    out = []
    for graphs in (1, 0):
        ctx = context(lbib, body, prec)
        lbib.lbib_set_graphs(ctx.h, graphs)
        lbib.lbib_set_output(ctx.h, every)
        got = []
        for k in calls:
            ctx.step(k)
            got += list(ctx.fields())
        got.append(ctx.populations())
        out.append((got, ctx.counters()[0]))
        ctx.close()
    assert out[0][1] == out[1][1] == sum(calls)
    for a, b in zip(out[0][0], out[1][0]):
        if body:
            assert np.abs(a - b).max() < 1e-13 * np.abs(b).max()
        else:
            assert np.array_equal(a, b)
