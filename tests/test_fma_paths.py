"""The arithmetic forms the kernels use in place of the definitions, re-derived
on the CPU: the quantiser and the own-code dequantiser as one float32 fused
multiply-add each, the first two micro-rotations of the row pass as one linear
map, and the transposed rotations on signed, offset operands (one shift-add
per half micro-rotation).  A GPU case runs tables that mix entries with and
without an exact float multiplier through every forward entry point."""
import numpy as np
import pytest

from oracle import codec, cordic_loeffler as cl, ijg, interval

MAGIC = 12582912.0                      # 1.5 * 2^23
NS = (4, 5, 6)
Y_MAX = 719380                          # largest |node| of the forward graph


def test_node_bound_covers_the_quantiser_range():
    for n in NS:
        assert interval.forward_bounds(sig=cl.Sigmas(n))[1] <= Y_MAX


def float_multiplier(m):
    """M * 2^-32 in float32 (the next float up where exact halves can occur), or None."""
    if int(np.float32(m)) != m:
        return None
    f = np.float32(m * 2.0 ** -32)
    return np.nextafter(f, np.float32(1)) if (m & 0xFFF) == 0 else f


@pytest.mark.parametrize("n", NS)
def test_fma_quantiser_equals_the_definition(n):
    """Every reachable multiplier over every |Y|: the product is exact in
    float64 (20 + 24 bits), so rint is the fused multiply-add's rounding."""
    y = np.arange(0, Y_MAX + 1, dtype=np.int64)
    yd = y.astype(np.float64)
    qs = range(1, 256) if n == 6 else [1, 2, 3, 4, 5, 7, 8, 16, 31, 32, 64, 99, 128, 254, 255]
    inexact, seen = set(), set()
    for q in qs:
        for m in np.unique(codec.quant_multipliers(np.full(64, q), n).astype(np.int64)):
            m = int(m)
            if m in seen:
                continue
            seen.add(m)
            f = float_multiplier(m)
            if f is None:
                inexact.add(q)
                continue
            assert np.array_equal(np.rint(yd * float(f)).astype(np.int64), (y * m + (1 << 31)) >> 32), (q, m)
    assert inexact <= {1, 2}            # only the finest steps fall back to the integer form


@pytest.mark.parametrize("n", NS)
def test_fma_dequantiser_is_exact(n):
    w = np.unique(codec.dequant_weights(n).astype(np.int64))
    for q in range(1, 256):
        for ww in w:
            qw = int(q * ww)
            c = MAGIC * (1 - qw)
            assert float(np.float32(qw)) == qw and float(np.float32(c)) == c
            lim = 1219 // q              # this library's own codes keep |q Q| < 1220
            for code in (-lim, -1, 0, 1, lim):
                exact = (MAGIC + code) * qw + c
                assert exact == MAGIC + code * qw and abs(code * qw) < 1 << 22


@pytest.mark.parametrize("n", NS)
def test_row_pass_steps_1_and_2_are_linear(n):
    rng = np.random.default_rng(n)
    for sig in (cl.Sigmas(n).odd_upper, cl.Sigmas(n).odd_lower, cl.Sigmas(n).even):
        a, b = rng.integers(-1100, 1101, size=(2, 2000)) * 16
        x, y = cl.cordic_rotate(a, b, sig[:2])
        c, k = 1 - sig[0] * sig[1] / 8, sig[0] / 2 + sig[1] / 4
        assert np.array_equal(x, a * c + b * k) and np.array_equal(y, b * c - a * k)


def offset_run(sig, ka, kb, upto):
    """Offsets and signs after `upto` transposed steps from (+a + ka, +b + kb); None when a shift is not exact."""
    sa = sb = 1
    for i in range(1, upto + 1):
        s, m = -sig[i - 1], 1 << i
        if (kb if sb > 0 else kb + 1) % m or (ka if sa > 0 else ka + 1) % m:
            return None
        cb = kb // m if sb > 0 else (kb + 1) // m - 1
        ca = ka // m if sa > 0 else (ka + 1) // m - 1
        fa, fb = sb != sa * s, sa != -s * sb
        ka, kb = (-ka if fa else ka) + cb, (-kb if fb else kb) + ca
        sa, sb = (-sa if fa else sa), (-sb if fb else sb)
    return ka, kb, sa, sb


@pytest.mark.parametrize("n", NS)
@pytest.mark.parametrize("name", ["odd_upper", "odd_lower", "even"])
def test_offset_rotation_equals_the_transposed_rotation(n, name):
    sig = getattr(cl.Sigmas(n), name)
    ka = kb = bits = 0
    for i in range(1, n + 1):                                # lift the starting offsets step by step
        sol = [(x, y) for x in range(1 << i) for y in range(1 << i)
               if offset_run(sig, ka + (x << bits), kb + (y << bits), i) is not None]
        assert len(sol) == 1                                 # exactly one solution modulo 2^(1 + .. + i)
        ka, kb, bits = ka + (sol[0][0] << bits), kb + (sol[0][1] << bits), bits + i
    m = 1 << bits
    ka, kb = (ka - m if ka >= m // 2 else ka), (kb - m if kb >= m // 2 else kb)
    eka, ekb, esa, esb = offset_run(sig, ka, kb, n)
    assert max(map(abs, (ka, kb, eka, ekb))) < 1 << 22       # nodes below 1.17e9 leave room in int32
    rng = np.random.default_rng(10 * n)
    lim = 1 << 29
    a = np.concatenate([rng.integers(-lim, lim, 5000), rng.integers(-70, 71, 5000), [-lim, lim, 0, -1, 1]])
    b = np.concatenate([rng.integers(-lim, lim, 5000), rng.integers(-70, 71, 5000), [lim, -lim, 0, 1, -1]])
    A, B, sa, sb = a + ka, b + kb, 1, 1
    for i in range(1, n + 1):
        s = -sig[i - 1]
        fa, fb = sb != sa * s, sa != -s * sb
        A, B = ((B >> i) - A if fa else A + (B >> i)), ((A >> i) - B if fb else B + (A >> i))
        assert max(np.abs(A).max(), np.abs(B).max()) < 1 << 31
        sa, sb = (-sa if fa else sa), (-sb if fb else sb)
    wa, wb = cl.cordic_rotate_t(a, b, sig)
    assert np.array_equal(A, esa * wa + eka) and np.array_equal(B, esb * wb + ekb)


@pytest.mark.gpu
@pytest.mark.parametrize("n", NS)
@pytest.mark.parametrize("steps", [[1] * 64, [2] * 64, [3] * 64, [1, 2, 3, 4] * 16, [255] * 32 + [1] * 32])
def test_tables_around_the_exact_multiplier_limit(cuda_ok, n, steps):
    """Q = 1 and 2 reach past a float's 24 bits (integer form), Q >= 3 never; images whose last tile and
    half tile are partly filled."""
    import torch

    from paper_1306_1373_gb300 import dctgb as D
    rng = np.random.default_rng(sum(steps) + n)
    imgs = [rng.integers(0, 256, size=s, dtype=np.uint8) for s in ((8, 8), (24, 8 * 17), (40, 8 * 33), (13, 301))]
    q = np.array(steps).reshape(8, 8)
    with D.cordic_variant(n):
        t = [torch.from_numpy(i).cuda() for i in imgs]
        want = [codec.compress_plane(i, q, n) for i in imgs]
        wrec = [codec.reconstruct_plane(c, q, *i.shape, n=n) for c, i in zip(want, imgs)]
        codes = np.concatenate([c.reshape(-1) for c in want])
        with D.Plan(512, 64, max_batch=4) as plan:
            assert np.array_equal(D.dct_compress(plan, t, 0, qtab=q).cpu().numpy(), codes)
            rec = [torch.zeros_like(x) for x in t]
            out = torch.zeros(codes.size, dtype=torch.int16, device="cuda")
            D.dct_codec_fused(plan, t, 0, qtab=q, coeffs=out, recon_planes=rec)
            assert np.array_equal(out.cpu().numpy(), codes)
            assert all(np.array_equal(r.cpu().numpy(), w) for r, w in zip(rec, wrec))
            for lanes in (1, 2):
                sizes = [c.size for c in want]
                out.zero_()
                rec = [torch.zeros_like(x) for x in t]
                items = D.make_batch_items(t, [0] * 4, coeffs=list(out.split(sizes)), recons=rec, qtabs=[q] * 4)
                for ops in (D.DCT_OP_COMPRESS | D.DCT_OP_RECONSTRUCT,
                            D.DCT_OP_COMPRESS | D.DCT_OP_RECONSTRUCT | D.DCT_OP_TWO_PASS):
                    out.zero_()
                    D.dct_batch_prepare(plan, items, ops, shape=(64, 2, 32, lanes))
                    D.dct_batch_launch(plan)
                    assert np.array_equal(out.cpu().numpy(), codes)
                    assert all(np.array_equal(r.cpu().numpy(), w) for r, w in zip(rec, wrec))


@pytest.mark.gpu
@pytest.mark.parametrize("quality", [92, 93, 100])
def test_rgb_at_the_exact_multiplier_limit(cuda_ok, quality):
    import torch

    from oracle import color
    from paper_1306_1373_gb300 import dctgb as D
    rgb = np.random.default_rng(quality).integers(0, 256, size=(37, 290, 3), dtype=np.uint8)
    with D.Plan(512, 64, layout=D.DCT_LAYOUT_YUV420) as plan:
        got = D.dct_compress_rgb(plan, torch.from_numpy(rgb).cuda(), quality).cpu().numpy()
    tabs = [ijg.luma_table(quality)] + [ijg.chroma_table(quality)] * 2
    want = np.concatenate([codec.compress_plane(p, t).reshape(-1) for p, t in zip(color.rgb_to_yuv420(rgb), tabs)])
    assert np.array_equal(got, want)
