"""The FP32 network's kernels at batch sizes where their splits have edges:
partial blocks of 8 and 16 rows, one and eleven gradient splits, ragged
32-row stages, the switch to 16 rows a block; and inputs off 16-byte
alignment."""
import numpy as np
import pytest

import oracle as O
from synth import params as SP

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_10521_gb300 as P
    c = P.Context(0)
    yield c
    torch.cuda.synchronize()
    c.close()


@pytest.mark.parametrize("B", [1, 7, 8, 33, 352, 353, 1023, 2433])
def test_gradients_and_forward(ctx, B):
    mlp = ctx.mlp_create(0)
    p = SP.mlp_params(21)
    ctx.mlp_set_params(mlp, p)
    X, T = SP.features(22, B), SP.targets(23, B)
    y_ref, _ = O.mlp_forward(p.astype(np.float64), X.astype(np.float64))
    loss_ref, g_ref = O.mlp_loss_grad(p.astype(np.float64), X.astype(np.float64), T.astype(np.float64))
    # FP32 dot products of 524 + 3 * 128 terms: a few 1e-6 of the activations' size; the logits here are of
    # order 1, so 1e-5 of the fraction; the gradients carry that through three more products
    assert np.max(np.abs(ctx.mlp_forward(mlp, X, half=False) - y_ref)) <= 1e-5
    g, loss = ctx.mlp_gradients(mlp, X, T)
    assert abs(loss - loss_ref) <= 1e-4 * loss_ref
    assert np.linalg.norm(g - g_ref) <= 1e-4 * np.linalg.norm(g_ref)
    mlp.free()


@pytest.mark.parametrize("B", [9, 130])
def test_unaligned_features(ctx, B):
    """Features that start off a 16-byte boundary take narrower copies, with the same sums."""
    import torch
    X = torch.from_numpy(SP.features(31, B)).cuda()
    T = torch.from_numpy(SP.targets(32, B)).cuda()
    room = torch.zeros(X.numel() + 1, device="cuda")
    odd = room[1:].view(X.shape)
    odd.copy_(X)
    out = []
    for x in (X, odd):
        mlp = ctx.mlp_create(0)
        ctx.mlp_set_params(mlp, SP.mlp_params(33))
        for _ in range(2):
            ctx.mlp_train_step(mlp, x, T, 1e-3)
        out += [ctx.mlp_params(mlp), ctx.mlp_forward(mlp, x, half=False).cpu().numpy(),
                ctx.mlp_forward(mlp, x, half=True).cpu().numpy()]
        mlp.free()
    for a, b in zip(out[:3], out[3:]):
        assert np.array_equal(a, b)
