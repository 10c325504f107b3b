"""The network without tensor maps (a driver that cannot encode them): its
products run one by one, against the FP64 oracle at the tolerances of
tests/test_gpu_network_sizes.py."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from tests.test_gpu_proposal import _batch, _bf16, _params, _rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 129, 1100])
def test_forward_gradients_and_update(n):
    import torch
    from paper_1807_02587_gb300 import binding as B
    p = _params(3)
    X, L = _batch(4, n)
    x, lab = _bf16(torch, X), torch.from_numpy(L).cuda()
    net = B.Mlp(n)
    B.hgmm_mlp_set_params(net.handle, p)
    B.hgmm_debug_mlp_maps(net.handle, False)
    y = torch.zeros((n, 9), dtype=torch.float32, device="cuda")
    B.hgmm_mlp_forward(net.handle, x, y)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    B.hgmm_mlp_gradients(net.handle, x, lab, n, w_t=2.0, loss=loss)
    B.hgmm_mlp_sync(net.handle)
    emu_y, _ = M.forward(p.astype(np.float64), X, act_bf16=True)
    assert _rel(y.cpu().numpy(), emu_y) < 1e-3
    g = B.hgmm_mlp_read_grads(net.handle)
    emu_loss, emu, _ = M.backward(p.astype(np.float64), X, L.astype(np.float64), 2.0, act_bf16=True)
    assert abs(loss.item() - emu_loss) < 1e-4 * emu_loss
    G, E = M.unpack(g.astype(np.float64)), M.unpack(emu)
    for name, _ in M.SHAPES:
        assert _rel(G[name], E[name]) < 2e-3, name
    idx = torch.arange(n, dtype=torch.int32, device="cuda")
    B.hgmm_mlp_train_step(net.handle, x, lab, n, index=idx, w_t=2.0, lr=1e-3, loss=loss)
    B.hgmm_mlp_sync(net.handle)
    assert np.array_equal(B.hgmm_mlp_read_grads(net.handle), g)
    w, _, _ = M.adam_step(p.astype(np.float64), g.astype(np.float64), 0.0, 0.0, 1, 1e-3)
    got = B.hgmm_mlp_get_params(net.handle).astype(np.float64)
    assert np.max(np.abs(got - w)) < 1e-6 * (1 + np.abs(w)).max()
