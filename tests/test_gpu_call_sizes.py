"""Direct calls of different sizes in any order, on two streams: the CTA size, the
grid and the kernel's shared-memory limit follow each call, not the one before."""
import numpy as np
import pytest
import torch

from oracle import codec, ijg, psnr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0, 2), (1, 2, 0, 1, 2)])
def test_small_and_large_calls_interleave(cuda_ok, order):
    from paper_1306_1373_gb300 import dctgb as D
    rng = np.random.default_rng(len(order))
    shapes = [(8, 8), (256, 640), (1096, 2056)]       # fewer tiles than SMs, a few per SM, several rounds
    imgs = [rng.integers(0, 256, size=s, dtype=np.uint8) for s in shapes]
    imgs = [np.minimum(i, 100 + (np.arange(i.shape[1]) % 90)).astype(np.uint8) for i in imgs]
    want = []
    for i in imgs:
        c = codec.compress_plane(i, ijg.luma_table(70))
        want.append((c.reshape(-1), psnr.sse(i, codec.reconstruct_plane(c, ijg.luma_table(70), *i.shape))))
    streams = [torch.cuda.Stream(), torch.cuda.current_stream()]
    with D.Plan(4096, 4096) as plan:
        for n, k in enumerate(order):
            t = torch.from_numpy(imgs[k]).cuda()
            torch.cuda.synchronize()
            with torch.cuda.stream(streams[n % 2]):
                codes = D.dct_compress(plan, [t], 70)
                stats = torch.zeros(1, D.STATS_WORDS, dtype=torch.int64, device="cuda")
                again = D.dct_compress(plan, [t], 70, stats=stats)
                out = torch.empty_like(t)
                sse = [D.dct_codec_fused(plan, [t], 70), D.dct_reconstruct(plan, codes, [out], 70, ref_planes=[t])]
                torch.cuda.synchronize()
            assert np.array_equal(codes.cpu().numpy(), want[k][0]) and torch.equal(codes, again)
            assert [int(s[0]) for s in sse] == [want[k][1]] * 2
            assert int(stats[0, 64]) == int(np.pad(imgs[k], [(0, -s % 8) for s in imgs[k].shape], mode="edge").sum())
