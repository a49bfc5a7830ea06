"""A network launch whose tensor-core wait gives up ends after that one wait:
its clean-up waits for nothing that was never issued."""
import time

import numpy as np
import pytest

from synth import params as SP

pytestmark = pytest.mark.gpu

WAIT = 0.25      # seconds after which a wait gives up


@pytest.mark.parametrize("rows", [1, 129])
def test_giving_up_takes_one_wait(rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_10521_gb300 as P
    ctx = P.Context(0)
    mlp = ctx.mlp_create(0)
    X = SP.features(12, rows)
    want = ctx.mlp_forward(mlp, X, half=True)
    ctx.test_inject(1)           # the first group of MMAs is neither issued nor committed
    t0 = time.perf_counter()
    with pytest.raises(P.ObbError) as e:
        ctx.mlp_forward(mlp, X, half=True)
    spent = time.perf_counter() - t0
    assert e.value.code == -6
    assert WAIT <= spent < 1.6 * WAIT
    assert np.array_equal(ctx.mlp_forward(mlp, X, half=True), want)
    mlp.free()
    ctx.close()
