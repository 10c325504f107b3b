"""The weight gradients' sums over the batch, apart from the BF16 storage of
their operands: the parameters here (one power of two per row or column) make
every hidden activation and every backward signal a value that BF16 holds
exactly, so dW1 = dZ1^T X, dW2 = dZ2^T H1 and dW3 = dY^T H2 differ from float64
only by the FP32 sums of the tensor core.

Bounds: the tensor core rounds its running FP32 sum towards zero at every
16-row step (at most 2^-23 of it, 2^-24 on average).  Of a sum of s steps that
grows evenly, each step's sum is on average half the last, so the error is
about s / 2 * 2^-24; the sums over accumulators and K slices, rounded to
nearest, add about 2^-24.  4,096 rows with at most 1/16 (dW1) and 1/32 (dW2,
dW3) of the batch per accumulator: s = 16 and 8, 5.4e-7 and 3.0e-7 for terms of
one sign; these terms have both signs and cancel to about half their size on
average, which random-sign rounding of a running sum near half its final size
does not follow: half the figures, 2.7e-7 and 1.5e-7, is the expectation, and
a third more the bound.  (Accumulators of 1/8 of the batch would give 5.4e-7.)
"""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from tests.test_gpu_proposal import _bf16

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def exact_params(rng):
    W1, W2, W3 = np.zeros((256, 1280)), np.zeros((256, 256)), np.zeros((9, 256))
    W1[np.arange(256), rng.choice(1280, 256, replace=False)] = 2.0 ** rng.integers(-1, 2, 256)
    W2[np.arange(256), rng.permutation(256)] = 2.0 ** rng.integers(-1, 2, 256)
    W3[rng.integers(0, 9, 256), np.arange(256)] = 2.0 ** rng.integers(-7, -4, 256) * rng.choice([-1, 1], 256)
    p = M.pack({"W1": W1, "b1": np.zeros(256), "W2": W2, "b2": np.zeros(256), "W3": W3,
                "b3": np.array([1, 0, 0, 0, 1, 0, 0, 0, 0.0])})
    return p.astype(np.float32), W1, W2, W3


# batch sizes: one 64-row chunk per accumulator, accumulators left unused, a
# ragged last chunk, every accumulator of every slice in use
@pytest.mark.parametrize("n, bounds", [(64, (1.8e-7,) * 3), (700, (1.8e-7,) * 3), (1025, (1.8e-7,) * 3),
                                       (4096, (3.6e-7, 2.0e-7, 2.0e-7))])
def test_sums_against_float64(n, bounds):
    import torch
    from paper_1807_02587_gb300 import binding as B
    rng = np.random.default_rng(7)
    p, W1, W2, W3 = exact_params(rng)
    # features as trees have them: weights -log u >= 0, means and covariances of both signs
    X = rng.normal(size=(n, 128, 10)) * 0.5
    X[..., 0] = -np.log(rng.random((n, 128)) + 1e-6)
    X = M.bf16((X * (rng.random((n, 128, 1)) > 0.25)).reshape(n, 1280))
    L = np.concatenate([np.tile(np.eye(3).ravel(), (n, 1)), np.zeros((n, 3))], axis=1) + 0.1 * rng.normal(size=(n, 12))
    L = L.astype(np.float32)
    net = B.Mlp(n)
    B.hgmm_mlp_set_params(net.handle, p)
    x, lab = _bf16(torch, X), torch.from_numpy(L).cuda()
    y = torch.zeros((n, 9), dtype=torch.float32, device="cuda")
    B.hgmm_mlp_forward(net.handle, x, y)
    B.hgmm_mlp_gradients(net.handle, x, lab, n)
    B.hgmm_mlp_sync(net.handle)
    G = M.unpack(B.hgmm_mlp_read_grads(net.handle).astype(np.float64))
    H1 = np.maximum(X @ W1.T, 0.0)
    H2 = np.maximum(H1 @ W2.T, 0.0)
    assert np.array_equal(M.bf16(H1), H1) and np.array_equal(M.bf16(H2), H2)
    dY = M.bf16(M.loss_grad(y.cpu().numpy().astype(np.float64), L.astype(np.float64), 1.0))
    dZ2 = (dY @ W3) * (H2 > 0)
    dZ1 = (dZ2 @ W2) * (H1 > 0)
    assert np.array_equal(M.bf16(dZ2), dZ2) and np.array_equal(M.bf16(dZ1), dZ1)
    ref = {"W1": dZ1.T @ X, "W2": dZ2.T @ H1, "W3": dY.T @ H2}
    got = {k: _rel(G[k], r) for k, r in ref.items()}
    print(n, got)
    for (k, e), b in zip(got.items(), bounds):
        assert e < b, (k, e, b)
