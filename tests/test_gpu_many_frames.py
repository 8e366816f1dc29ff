"""Features and inference over many frames: every launch shape that the number
of frames selects gives the bits of the calls on a few frames at a time."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FEATURE_SIZES = [1, 31, 33, 16500, 1 << 17, (1 << 18) + 1]     # 20, 15, 2 and 1 groups of features


@pytest.mark.parametrize("n", FEATURE_SIZES)
def test_features_do_not_depend_on_the_number_of_frames(cuda_ok, n):
    import torch

    from paper_1306_1373_gb300 import dctgb as D
    rng = np.random.default_rng(n)
    st = torch.from_numpy(rng.integers(1, 1 << 40, size=(n, D.STATS_WORDS))).cuda()
    w, h = (torch.from_numpy(rng.integers(8, 4097, n).astype(np.int32)).cuda() for _ in range(2))
    t = torch.from_numpy(rng.uniform(25, 45, n).astype(np.float32)).cuda()
    got = D.dct_features(st, w, h, t)
    for a in sorted({0, n // 2, max(0, n - 40)}):
        s = slice(a, min(n, a + 40))
        assert torch.equal(got[s], D.dct_features(st[s].contiguous(), w[s].contiguous(), h[s].contiguous(), t[s].contiguous()))


@pytest.mark.parametrize("n", [4863, 4864, 4865, 4866, 4867, 1024 * 32 + 1, 3 * 1024 * 32 - 2])
@pytest.mark.parametrize("bf16", [True, False])
def test_inference_does_not_depend_on_the_number_of_samples(cuda_ok, n, bf16):
    import torch

    from paper_1306_1373_gb300 import dctgb as D, rc
    f = torch.from_numpy(np.random.default_rng(n).normal(0, 2, size=(n, 80)).astype(np.float32)).cuda()
    net = D.Mlp(rc.init_params(4), act_bf16=bf16)
    net.set_norm(f)
    y, q = net.forward(f)
    part = [net.forward(f[a:a + 4000]) for a in range(0, n, 4000)]
    assert torch.equal(y, torch.cat([p[0] for p in part])) and torch.equal(q, torch.cat([p[1] for p in part]))
