"""Direct calls captured into a CUDA graph: the calls that clear words and launch
the kernel behind the clear as a programmatic dependent give, on every replay,
what the same calls give outside, also back to back on the same words."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(8, 8), (40, 301), (512, 640)])
def test_direct_calls_replay(cuda_ok, size):
    import torch

    from paper_1306_1373_gb300 import dctgb as D
    rng = np.random.default_rng(size[1])
    img = torch.zeros(size, dtype=torch.uint8, device="cuda")
    codes, fcodes = (torch.zeros(D.coeff_count([size]), dtype=torch.int16, device="cuda") for _ in range(2))
    rec, frec, erec = (torch.zeros_like(img) for _ in range(3))
    st = torch.zeros(1, D.STATS_WORDS, dtype=torch.int64, device="cuda")
    sse, fsse, esse = (torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(3))
    out = {}

    def calls(plan):
        for _ in range(2):                       # the second clear follows the first kernel's sums
            D.dct_compress(plan, [img], 75, coeffs=codes, stats=st)
            D.dct_reconstruct(plan, codes, [rec], 75, ref_planes=[img], sse=sse)
            D.dct_codec_fused(plan, [img], 75, coeffs=fcodes, recon_planes=[frec], sse=fsse)
            D.dct_exact_fused(plan, [img], 75, recon_planes=[erec], sse=esse)
            out["entropy"] = D.dct_entropy_stats(plan, codes, [size])

    def results():
        return [t.clone() for t in (codes, fcodes, rec, frec, erec, st, sse, fsse, esse, out["entropy"])]

    with D.Plan(*size[::-1]) as plan:
        calls(plan)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            calls(plan)
        entropy = out["entropy"]
        for seed in range(3):
            img.copy_(torch.from_numpy(rng.integers(0, 256, size=size, dtype=np.uint8)))
            for t in (codes, fcodes, rec, frec, erec, st, sse, fsse, esse):
                t.fill_(7)
            out["entropy"] = entropy
            graph.replay()
            got = results()
            calls(plan)
            assert all(torch.equal(a, b) for a, b in zip(got, results())), seed
            assert torch.equal(got[0], got[1]) and torch.equal(got[6], got[7])
        torch.cuda.synchronize()
