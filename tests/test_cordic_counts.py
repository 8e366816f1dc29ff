"""CORDIC counts without a library of their own in the default build, which
cordic_variant builds on demand: past 6 the forward graph runs in integers and
the transposed rotations carry no offsets."""
import subprocess

import numpy as np
import pytest

from oracle import codec, ijg
from paper_1306_1373_gb300 import build
from test_fma_paths import cl, offset_run

NAMES = ("odd_upper", "odd_lower", "even")


@pytest.mark.parametrize("n", [3, 4, 6, 7, 8])
def test_offsets_of_the_transposed_rotations(tmp_path, n):
    src = tmp_path / "offsets.cu"
    src.write_text('#include <cstdio>\n#include "kernels.cuh"\nusing namespace dctgb;\ntemplate <unsigned M> void show() { using R = TrRotation<M>; '
                   'printf("%lld %lld %lld %lld %d %d\\n", R::start.a, R::start.b, R::end.ka, R::end.kb, R::end.sa, R::end.sb); }\n'
                   'int main() { show<kSigOddUpper>(); show<kSigOddLower>(); show<kSigEven>(); }\n')
    exe = str(tmp_path / "offsets")
    subprocess.run([build._nvcc()] + build.ARCH + ["-std=c++17", "-DDCTGB_CORDIC_N=%d" % n, "-I" + build.INCLUDE, "-I" + build.CSRC,
                                                   "-o", exe, str(src)], check=True, capture_output=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    for name, line in zip(NAMES, lines):
        ka, kb, *end = map(int, line.split())
        if n > 6:
            assert [ka, kb] + end == [0, 0, 0, 0, 1, 1], name       # the plain form
        else:
            assert offset_run(getattr(cl.Sigmas(n), name), ka, kb, n) == tuple(end), name


@pytest.mark.gpu
@pytest.mark.parametrize("n", [7])
def test_calls_match_the_oracle_at_n(cuda_ok, n):
    import torch

    from paper_1306_1373_gb300 import dctgb as D
    rng = np.random.default_rng(n)
    imgs = [rng.integers(0, 256, size=s, dtype=np.uint8) for s in ((8, 8), (40, 301), (128, 264))]
    imgs.append(((np.indices((64, 64)).sum(0) & 1) * 255).astype(np.uint8))
    with D.cordic_variant(n):
        t = [torch.from_numpy(i).cuda() for i in imgs]
        for quality in (20, 75, 96):
            tab = ijg.luma_table(quality)
            want = [codec.compress_plane(i, tab, n) for i in imgs]
            wrec = [codec.reconstruct_plane(c, tab, *i.shape, n=n) for c, i in zip(want, imgs)]
            codes = np.concatenate([c.reshape(-1) for c in want])
            with D.Plan(512, 512, max_batch=4) as plan:
                out = torch.zeros(codes.size, dtype=torch.int16, device="cuda")
                rec = [torch.zeros_like(x) for x in t]

                def check():
                    assert np.array_equal(out.cpu().numpy(), codes)
                    assert all(np.array_equal(r.cpu().numpy(), w) for r, w in zip(rec, wrec))

                D.dct_compress(plan, t, quality, coeffs=out)
                D.dct_reconstruct(plan, out, rec, quality)
                check()
                out.zero_()
                [r.zero_() for r in rec]
                D.dct_codec_fused(plan, t, quality, coeffs=out, recon_planes=rec)
                check()
                items = D.make_batch_items(t, [quality] * 4, coeffs=list(out.split([c.size for c in want])), recons=rec)
                ops = D.DCT_OP_COMPRESS | D.DCT_OP_RECONSTRUCT
                for lanes in (1, 2):
                    for extra in (0, D.DCT_OP_TWO_PASS):
                        out.zero_()
                        [r.zero_() for r in rec]
                        D.dct_batch_prepare(plan, items, ops | extra, shape=(64, 2, 32, lanes))
                        D.dct_batch_launch(plan)
                        check()
