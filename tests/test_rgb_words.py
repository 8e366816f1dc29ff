"""RGB conversion four pixels at a time (word loads, 16-bit products of
complemented bytes): the integers on the CPU over every colour, and the codes of
dct_compress_rgb on the GPU at every byte offset of the rows and at widths
around a group of four pixels and a strip of 256."""
import numpy as np
import pytest
import torch

from oracle import codec, color, ijg


def test_complemented_products_equal_the_conversion():
    g, b = np.meshgrid(np.arange(256), np.arange(256), indexing="ij")
    for r in range(256):
        rgb = np.stack([np.full_like(g, r), g, b], axis=-1)
        cb = 11058 * (255 - r) + 21710 * (255 - g) + 32768 * b + 65536
        cr = 32768 * r + 27439 * (255 - g) + 5329 * (255 - b) + 65536
        y = 19595 * r + 38470 * g + 7471 * b + 32768
        assert max(y.max(), cb.max(), cr.max()) < 2 ** 32
        want = color.rgb_to_yuv420(np.repeat(np.repeat(rgb.astype(np.uint8), 2, 0), 2, 1))
        assert np.array_equal(y >> 16, want[0][::2, ::2])
        # a 2x2 quad of one colour averages to that colour's chroma
        assert np.array_equal(np.minimum(cb >> 16, 255), want[1])
        assert np.array_equal(np.minimum(cr >> 16, 255), want[2])


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 1, 2, 3, 5, 14, 15])
@pytest.mark.parametrize("w", [2, 3, 4, 5, 254, 255, 256, 257, 260])
def test_codes_at_every_row_offset(cuda_ok, offset, w):
    from paper_1306_1373_gb300 import dctgb as D
    h = 19
    rng = np.random.default_rng(100 * w + offset)
    rgb = rng.integers(0, 256, size=(h, w, 3), dtype=np.uint8)
    rgb[rng.random((h, w)) < 0.3] = [255, 0, 255]
    rgb[rng.random((h, w)) < 0.2] = [0, 255, 0]
    pitch = 3 * w + 1                                     # the offset moves from row to row
    buf = torch.zeros(offset + h * pitch, dtype=torch.uint8, device="cuda")
    view = torch.as_strided(buf, (h, w, 3), (pitch, 3, 1), storage_offset=offset)
    view.copy_(torch.from_numpy(rgb))
    with D.Plan(512, 512) as plan:
        codes = D.dct_compress_rgb(plan, view, 95)
        torch.cuda.synchronize()
    planes = color.rgb_to_yuv420(rgb)
    tabs = (ijg.luma_table(95), ijg.chroma_table(95), ijg.chroma_table(95))
    want = np.concatenate([codec.compress_plane(p, q).reshape(-1) for p, q in zip(planes, tabs)])
    assert np.array_equal(codes.cpu().numpy(), want)
