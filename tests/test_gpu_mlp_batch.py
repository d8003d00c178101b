"""The schedule network's kernels at the edges of their blocks (16 samples per block,
eight blocks per gradient): gradient, loss and outputs against the fp64 oracle of the
same bf16-rounded weights, and the one-launch training loop against its steps taken
one by one through the gradient and Adam entry points."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_1709_04394_gb300 import gbmc
from tests.gpu_common import ctx, torch  # noqa: F401

pytestmark = pytest.mark.gpu


def _inputs(n, seed):
    rng = np.random.default_rng(seed)
    p = (rng.uniform(-1, 1, omlp.N_PARAMS) / 8).astype(np.float32)
    X = rng.uniform(-1.5, 1.5, (n, 6)).astype(np.float32)
    T = rng.normal(-0.5, 0.4, n).astype(np.float32)
    return p, X, T


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("B", [1, 15, 16, 17, 100, 127, 128])
def test_gradient_at_block_edges(ctx, B):
    p, X, T = _inputs(B, B)
    g = torch.full((omlp.N_PARAMS,), 7.0, device="cuda")
    loss = torch.zeros(1, device="cuda")
    gbmc.mlp_grad(ctx, _dev(p), _dev(X), _dev(T), g, loss)
    pb, X64, T64 = omlp.bf16_round(p), X.astype(np.float64), T.astype(np.float64)
    ref = omlp.grad(pb, X64, T64)
    # fp32 products and sums of at most 128 + 64 terms of order max|g|: 200 * 2^-24 = 1.2e-5
    np.testing.assert_allclose(g.cpu().numpy(), ref, rtol=1e-4, atol=1.2e-5 * np.abs(ref).max())
    assert float(loss) == pytest.approx(omlp.loss(pb, X64, T64), rel=1e-5)


@pytest.mark.parametrize("B", [1, 16, 17, 1517, 20000])
def test_outputs_at_block_edges(ctx, B):
    p, X, _ = _inputs(B, B + 1)
    Y = torch.zeros(B, device="cuda")
    gbmc.mlp_forward(ctx, _dev(p), _dev(X), Y)
    ref, _ = omlp.forward(omlp.bf16_round(p), X.astype(np.float64))
    # sums of 70 fp32 terms of order 1 through two layers: 140 * 2^-24 = 8.3e-6
    np.testing.assert_allclose(Y.cpu().numpy(), ref, rtol=0, atol=1e-5)


@pytest.mark.parametrize("n,batch,epochs", [(100, 32, 2), (16, 128, 3), (300, 1, 1)])
def test_training_equals_single_steps(ctx, n, batch, epochs):
    # (300 steps of one sample: more than one launch)
    p0, X, T = _inputs(n, 3)
    X, T = _dev(X), _dev(T)
    nb = -(-n // batch)
    losses = torch.zeros(epochs * nb, device="cuda")
    p = _dev(p0)
    gbmc.mlp_train(ctx, p, X, T, epochs, batch, 1e-4, losses)
    q, m, v = _dev(p0), torch.zeros(omlp.N_PARAMS, device="cuda"), torch.zeros(omlp.N_PARAMS, device="cuda")
    g, loss, ref = torch.zeros(omlp.N_PARAMS, device="cuda"), torch.zeros(1, device="cuda"), []
    for k in range(epochs * nb):
        a = k % nb * batch
        gbmc.mlp_grad(ctx, q, X[a:a + batch], T[a:a + batch], g, loss)
        gbmc.mlp_adam(ctx, q, g, m, v, k + 1, 1e-4)
        ref.append(float(loss))
    # the same operations; a fused multiply-add placed otherwise moves an update by
    # 2^-22 of lr, which may round a weight to the other bf16 neighbour (2^-9 of its share)
    np.testing.assert_allclose(p.cpu().numpy(), q.cpu().numpy(), rtol=0, atol=1e-6)
    np.testing.assert_allclose(losses.cpu().numpy(), ref, rtol=1e-4)
