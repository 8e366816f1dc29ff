"""The float32 forms of the exact-DCT kernel, checked on the CPU: its seven
basis magnitudes reproduce the rounded FP64 basis, and its quotient (one
product with the rounded reciprocal and one residual step) is the correctly
rounded one; the rate kernel on codes that stress its walk."""
import math
import os
import re

import numpy as np
import pytest

HDR = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                        "paper_1306_1373_gb300", "csrc", "exact.cu")).read()


def test_basis_magnitudes_and_signs():
    mags = [np.float32(v) for v in re.findall(r"(\d\.\d+)f", HDR[HDR.index("mag[8]"):HDR.index("return mag[m]")])]
    assert len(mags) == 8
    for u in range(8):
        for i in range(8):
            c = np.float32(math.sqrt(2.0 / 8) * (1 / math.sqrt(2.0) if u == 0 else 1.0)
                           * math.cos(math.pi * u * (2 * i + 1) / 16.0))
            j = (u * (2 * i + 1)) % 32
            j = 32 - j if j > 16 else j
            m = 4 if u == 0 else (-(16 - j) if j > 8 else j)
            assert (-1 if m < 0 else 1) * mags[abs(m)] == c, (u, i)


def test_quotient_is_correctly_rounded():
    rng = np.random.default_rng(0)
    f = np.float32
    for q in range(1, 256):
        x = np.concatenate([rng.uniform(0, 1100, 40000), rng.integers(0, 2200, 4000) * q * 0.5,
                            10 ** rng.uniform(-8, 3, 4000)]).astype(f)
        r = f(1) / f(q)
        q0 = x * r
        res = (x.astype(np.float64) - np.float64(q) * q0.astype(np.float64)).astype(f)
        got = (res.astype(np.float64) * np.float64(r) + q0.astype(np.float64)).astype(f)
        assert np.array_equal(got, x / f(q)), q


@pytest.mark.gpu
@pytest.mark.parametrize("shapes", [[(8, 8)], [(8, 8 * 31)], [(8, 8 * 32)], [(8, 8 * 33)], [(72, 296), (8, 8), (16, 520)]])
@pytest.mark.parametrize("fill", ["zero", "last", "runs", "dense"])
def test_symbol_walk_on_designed_codes(cuda_ok, shapes, fill):
    """All-zero blocks, a lone value in the last zig-zag position (three ZRLs), runs of every length, no zeros."""
    import torch

    from oracle import entropy
    from paper_1306_1373_gb300 import dctgb as D
    rng = np.random.default_rng(len(fill) + len(shapes))
    total = sum(D.n_blocks(h, w) for h, w in shapes)
    q = np.zeros((total, 64), dtype=np.int16)
    if fill == "last":
        q[:, 63] = rng.integers(1, 1024, total)
    elif fill == "runs":
        q[np.arange(total), rng.integers(0, 64, total)] = rng.integers(-1023, 1024, total)
        q[np.arange(total), rng.integers(0, 64, total)] = -1
    elif fill == "dense":
        q[:] = np.where(rng.random(q.shape) < 0.5, 1, -1) * rng.integers(1, 1024, q.shape)
    with D.Plan(1024, 1024) as plan:
        st = D.dct_entropy_stats(plan, torch.from_numpy(q.reshape(-1)).cuda(), shapes).cpu().numpy()
    off = 0
    for row, (h, w) in zip(st, shapes):
        n = D.n_blocks(h, w)
        dc, ac, amp, nb = entropy.plane_histograms(q[off:off + n])
        assert row[:16].tolist() == dc and row[16:272].tolist() == ac and int(row[272]) == amp and int(row[273]) == nb
        off += n
