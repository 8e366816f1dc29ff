"""A training epoch (runs of steps in one cluster launch, or two launches a step
past batch 1024) gives the same bits as its steps made one by one with
dct_mlp_loss_grad and dct_mlp_adam."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(3, 1), (65, 63), (64, 64), (200, 65), (300, 256), (700, 257), (1000, 513),
                                     (2100, 1024), (2100, 1025)])
@pytest.mark.parametrize("bf16", [True, False])
def test_epoch_equals_single_steps(cuda_ok, n, batch, bf16):
    from paper_1306_1373_gb300 import dctgb as D, rc
    rng = np.random.default_rng(n + batch)
    feats = torch.from_numpy(rng.normal(3, 2, size=(n + 5, 80)).astype(np.float32)).cuda()
    labels = torch.from_numpy(rng.uniform(0, 1, n + 5).astype(np.float32)).cuda()
    order = torch.from_numpy(rng.permutation(n + 5)[:n].astype(np.int32)).cuda()
    nets = [D.Mlp(rc.init_params(1), act_bf16=bf16) for _ in range(2)]
    for net in nets:
        net.set_norm(feats)
    got, want = [], []
    for e in range(2):                       # the second epoch starts from used Adam state
        got.append(nets[0].train_epoch(feats, labels, order, batch=batch, lr=2e-3))
        for b0 in range(0, n, batch):
            loss, grad = nets[1].loss_grad(feats, labels, order[b0:b0 + batch].contiguous())
            nets[1].adam(grad, lr=2e-3)
            want.append(loss)
    assert nets[0].step == nets[1].step
    assert torch.equal(torch.cat(got), torch.cat(want))
    for a, b in ((nets[0].params, nets[1].params), (nets[0].m, nets[1].m), (nets[0].v, nets[1].v)):
        assert torch.equal(a, b)
