"""The number of steps by which lbib_batch_autotune advances the contexts, which a
caller that counts steps relies on: 20 * (24 + 12 * steps).
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


@pytest.mark.parametrize("steps", [1, 3])
def test_batch_autotune_advances_as_declared(lbib, steps):
    ctxs = [lbib.Context.from_case(W.case_empty(n=(12, 10 + k, 14), seed=k)) for k in range(2)]
    batch = lbib.Batch(ctxs)
    lbib.lbib_batch_autotune(batch.h, steps)
    assert batch.counters()[0] == 20 * (24 + 12 * steps)
    batch.close()
    for ctx in ctxs:
        assert ctx.counters()[0] == 20 * (24 + 12 * steps)
        ctx.close()
