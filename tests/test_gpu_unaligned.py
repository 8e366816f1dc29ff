"""Planes whose rows start at any address: word loads with funnel shifts and
split stores for the interior, byte access where a word would leave the plane.
Every call must give the aligned plane's results and write nothing outside
the output plane."""
import numpy as np
import pytest
import torch

from oracle import codec, ijg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D(cuda_ok):
    from paper_1306_1373_gb300 import dctgb
    dctgb.load()
    return dctgb


@pytest.mark.parametrize("w,h,pitch", [(8, 8, 8), (9, 16, 9), (16, 8, 17), (271, 24, 271), (264, 40, 266), (300, 16, 307)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3, 5])
def test_any_row_alignment(D, w, h, pitch, offset):
    rng = np.random.default_rng(w * 8 + offset)
    img = rng.integers(0, 256, size=(h, w), dtype=np.uint8)
    Q = ijg.luma_table(60)
    want = codec.compress_plane(img, Q)
    rec = codec.reconstruct_plane(want, Q, h, w)

    def plane(fill):
        buf = torch.full((offset + pitch * h + 16,), fill, dtype=torch.uint8, device="cuda")
        return buf, torch.as_strided(buf, (h, w), (pitch, 1), offset)

    _, src = plane(7)
    src.copy_(torch.from_numpy(img))
    codes = torch.empty(want.size, dtype=torch.int16, device="cuda")
    with D.Plan(512, 64, max_batch=1) as plan:
        runs = [lambda o: D.dct_codec_fused(plan, [src], 60, coeffs=codes, recon_planes=[o]),
                lambda o: D.dct_reconstruct(plan, D.dct_compress(plan, [src], 60, coeffs=codes), [o], 60, ref_planes=[src]),
                lambda o: D.dct_exact_fused(plan, [src], 60, recon_planes=[o])]
        for lanes in (1, 2):
            def graph(o, lanes=lanes):
                sse = torch.zeros(1, dtype=torch.int64, device="cuda")
                D.dct_batch_prepare(plan, D.make_batch_items([src], [60], coeffs=[codes], recons=[o]), 7, sse=sse,
                                    shape=(64, 1, 32, lanes))
                D.dct_batch_launch(plan)
                return sse
            runs.append(graph)
        for i, run in enumerate(runs):
            codes.zero_()
            buf, out = plane(201)
            sse = int(run(out)[0])
            got = out.cpu().numpy()
            if i != 2:
                assert np.array_equal(codes.cpu().numpy(), want.reshape(-1)) and np.array_equal(got, rec), i
            assert sse == int(((got.astype(np.int64) - img) ** 2).sum()), i
            mask = torch.ones_like(buf, dtype=torch.bool)
            torch.as_strided(mask, (h, w), (pitch, 1), offset).fill_(False)
            assert bool((buf[mask] == 201).all()), i
