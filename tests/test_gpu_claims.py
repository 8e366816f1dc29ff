"""What a warp of the two-lane batch kernels claims (half a tile, a tile, four
tiles) follows from the tiles per warp; on both sides of either limit, with
tiles whose second half is empty or partly filled, a graph gives the direct
calls' bytes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_warp,more", [(1, -1), (1, 0), (1, 1), (16, -1), (16, 0)])
@pytest.mark.parametrize("quality", [50, 96])
def test_graph_equals_direct_calls_around_the_claim_limits(cuda_ok, per_warp, more, quality):
    import torch

    from paper_1306_1373_gb300 import dctgb as D
    warps = 2 * torch.cuda.get_device_properties(0).multi_processor_count      # one CTA of 64 threads per SM
    ntiles = per_warp * warps + more
    sizes = [(8, 8), (8, 8 * 17), (24, 8 * 17), (5, 13)]                       # 1 + 1 + 2 + 1 tiles
    sizes.insert(2, (8 * (ntiles - 5), 256))                                   # a row of blocks is a tile
    rng = np.random.default_rng(ntiles)
    imgs = [torch.from_numpy(rng.integers(0, 256, size=s, dtype=np.uint8)).cuda() for s in sizes]
    with D.Plan(256, 65536, max_batch=len(imgs)) as plan:
        want = [torch.zeros(D.coeff_count([s]), dtype=torch.int16, device="cuda") for s in sizes]
        wrec = [torch.zeros_like(i) for i in imgs]
        wsse = torch.cat([D.dct_codec_fused(plan, [i], quality, coeffs=c, recon_planes=[r])
                          for i, c, r in zip(imgs, want, wrec)])
        C, R, S, T = D.DCT_OP_COMPRESS, D.DCT_OP_RECONSTRUCT, D.DCT_OP_SSE, D.DCT_OP_TWO_PASS
        for ops in (C | R | S, C | R | S | T, R | S, S):
            codes = [c.clone() if ops == (R | S) else torch.zeros_like(c) for c in want]
            rec = [torch.zeros_like(i) for i in imgs]
            sse = torch.full((len(imgs),), -1, dtype=torch.int64, device="cuda")
            items = D.make_batch_items(imgs, [quality] * len(imgs), codes, rec)
            D.dct_batch_prepare(plan, items, ops, sse=sse, shape=(64, 1, 32, 2))
            for _ in range(2):
                D.dct_batch_launch(plan)
            assert torch.equal(sse, wsse), ops
            if ops & C:
                assert all(map(torch.equal, codes, want)), ops
            if ops & R:
                assert all(map(torch.equal, rec, wrec)), ops
