"""The training cluster's exchange: no multicast load (the pointers a call gets
need not be memory of the launching GPU, and a multicast must read only that),
and no wait that polls memory (one that ran out would leave a half-trained
network behind).  Runs longer than one launch give the bits of single steps."""
import glob
import os

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1306_1373_gb300", "csrc")


@pytest.mark.parametrize("word", ["multicast::cluster", "mbarrier"])
def test_no_kernel_names(word):
    files = [f for ext in ("*.cu", "*.cuh", "*.h") for f in glob.glob(os.path.join(CSRC, ext))]
    assert files and not [f for f in files if word in open(f).read()]


@pytest.mark.gpu
@pytest.mark.parametrize("steps,batch,last", [(64, 64, 64), (65, 64, 1), (131, 64, 7), (66, 300, 257), (65, 1024, 700),
                                              (131, 1, 1), (70, 33, 5), (3, 5000, 4999)])
def test_epoch_of_several_launches(cuda_ok, steps, batch, last):
    import torch

    from paper_1306_1373_gb300 import dctgb as D, rc
    n = (steps - 1) * batch + last
    rng = np.random.default_rng(n)
    feats = torch.from_numpy(rng.normal(3, 2, size=(n, 80)).astype(np.float32)).cuda()
    labels = torch.from_numpy(rng.uniform(0, 1, n).astype(np.float32)).cuda()
    order = torch.from_numpy(rng.permutation(n).astype(np.int32)).cuda()
    nets = [D.Mlp(rc.init_params(2), act_bf16=True) for _ in range(2)]
    for net in nets:
        net.set_norm(feats)
    got = nets[0].train_epoch(feats, labels, order, batch=batch, lr=1e-3)
    want = []
    for b0 in range(0, n, batch):
        loss, grad = nets[1].loss_grad(feats, labels, order[b0:b0 + batch].contiguous())
        nets[1].adam(grad, lr=1e-3)
        want.append(loss)
    assert nets[0].step == nets[1].step == steps
    assert torch.equal(got, torch.cat(want))
    for a, b in ((nets[0].params, nets[1].params), (nets[0].m, nets[1].m), (nets[0].v, nets[1].v)):
        assert torch.equal(a, b)
