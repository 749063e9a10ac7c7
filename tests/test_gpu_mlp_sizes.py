"""The step network at sizes that fill no tile (products are tiled 32 x 32 x 32) against the FP64
oracle: loss and gradients to 1e-4 of the largest entry (FP32 sums of at most 600 terms)."""
import numpy as np
import pytest

from oracle import mlp as ref
from synth_inputs import mlp_init

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ni,nh,no,B", [(37, 70, 2, 1), (5, 3, 3, 65), (192, 96, 25, 513), (33, 32, 31, 600)])
def test_loss_gradients_and_forward(ni, nh, no, B):
    import torch
    import paper_2108_11989_gb300 as qs
    rng = np.random.default_rng(B)
    p0 = [p + np.float32(0.05) * rng.standard_normal(p.shape).astype(np.float32) for p in mlp_init(3, ni, nh, no)]
    X = rng.standard_normal((B, ni)).astype(np.float32)
    T = np.concatenate([rng.standard_normal((B, 1)), rng.random((B, no - 1)) < 0.3], axis=1).astype(np.float32)
    net = qs.MLP(ni, nh, no, max_batch=B)
    net.set_params(p0)
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    Y = net.forward(Xd).cpu().numpy()
    Yr, _ = ref.forward(p0, X)
    assert np.abs(Y - Yr).max() <= 1e-4 * np.abs(Yr).max()
    loss = net.train_step(Xd, Td, lr=1e-3)
    Lr, gr = ref.value_and_grad(p0, X, T)
    assert abs(loss - Lr) <= 1e-4 * abs(Lr)
    for g, h in zip(net.get_grads(), gr):
        assert np.abs(g - h).max() <= 1e-4 * np.abs(h).max() + 1e-7
    net.close()
