"""Bodies that move fast, in batches whose kernels are launched programmatically
one behind another and in a context alone: the kernels that begin before their
predecessor has ended read the positions of the step before.  The reference
is a context read (and so waited for) after every step.  Both differ only in
the order of the atomic spreading sums: 1e-10 as for recorded trajectories,
where a position one rotation of its three buffers old would be 0.1 off; FP32
1e-4 lattice units on positions and 1e-5 of the flow on velocities, doubled
because both sides carry the rounding.
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


UF = (0.06, -0.04, 0.05)


def cases(prec):
    out = []
    for k in range(10):
        n = (22 + k, 24, 21 + (k * 5) % 7)
        c = np.array([n[0] - 4.3, 3.7 + k, 10.21])
        z, y, x = np.meshgrid(*[np.arange(m) for m in n[::-1]], indexing="ij")
        u = np.zeros(z.shape + (3,)) + np.array(UF)
        u[..., 1] += 5e-3 * np.sin(2 * np.pi * x / n[0])
        v, f = W.icosphere(2, 4.0 + 0.1 * k, c)
        if k % 2:
            body = W.Body(v, f, rigid=True, density_ratio=1.3, ref_radius=4.0, u0=UF, omega0=(0.01, 0.02, -0.01))
        else:
            body = W.Body(v, f, ks0=2e-3, Eb=0.01, kv=1.0, ref_radius=4.0, mass_model=1)
        out.append(W.Case("moving%d" % k, n, 0.8, (0, 0, 0), np.zeros((6, 3)), precision=prec, bodies=[body],
                          u0=u.reshape(-1, 3)))
    return out


@pytest.mark.parametrize("how", ["batch", "alone", "persistent"])
@pytest.mark.parametrize("prec", [W.PREC_FP64, W.PREC_FP32])
def test_many_steps_at_once_equal_single_steps(lbib, prec, how):
    steps, todo = 27, cases(prec)
    ref = []
    for case in todo:
        ctx = lbib.Context.from_case(case)
        for _ in range(steps):
            ctx.step(1)
            ctx.markers(0)
        ref.append((ctx.markers(0), ctx.fields()[1]))
        ctx.close()
    ctxs = [lbib.Context.from_case(case) for case in todo]
    if how == "alone":
        for ctx in ctxs:
            ctx.step(steps)
    else:
        batch = lbib.Batch(ctxs)
        if how == "persistent":
            batch.set_persistent(1)
        batch.step(steps)
        batch.sync()
        batch.close()
    xtol, utol = (1e-10, 1e-10) if prec == W.PREC_FP64 else (2e-4, 2e-6)
    for ctx, case, ((X, V, F), u) in zip(ctxs, todo, ref):
        Xg, Vg, Fg = ctx.markers(0)
        assert np.abs(X - case.bodies[0].verts).max() > 1.0
        assert np.abs(Xg - X).max() < xtol
        assert np.abs(Vg - V).max() < utol
        assert np.abs(ctx.fields()[1] - u).max() < utol
        ctx.close()
