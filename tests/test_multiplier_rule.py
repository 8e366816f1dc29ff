"""The quantiser's multipliers at every quality step and CORDIC count: the
library's own rule for their float form, where exact halves can occur, and the
integer form of tables with a multiplier past a float's 24 bits."""
import subprocess

import numpy as np
import pytest

from oracle import codec
from paper_1306_1373_gb300 import build

Y_MAX = 719380                          # largest |node| of the forward graph
MAGIC_BITS = 0x4B400000
NS = (4, 5, 6)


def multipliers(n):
    return sorted({int(m) for q in range(1, 256) for m in np.ravel(codec.quant_multipliers(np.full(64, q), n))})


@pytest.mark.parametrize("n", NS)
def test_halves_occur_at_the_tie_entries_only(n):
    tie = np.zeros((8, 8), dtype=bool)
    tie[::4, ::4] = True
    for q in range(1, 256):
        m = codec.quant_multipliers(np.full(64, q), n).astype(np.int64).reshape(8, 8)
        assert (m[~tie] & 0xFFF).all()                          # |Y| < 2^20: no half (and a fitting M's float form is exact)
        assert (m[tie] == np.rint(2.0 ** 25 / q)).all()         # the same at every n


@pytest.mark.parametrize("n", NS)
def test_integer_form_on_float_bits(n):
    """High word of (bits - MAGIC_BITS) M + (MAGIC_BITS << 32) + 2^31 (less 1 for Y < 0 at the tie entries)."""
    y = np.arange(-Y_MAX, Y_MAX + 1, dtype=np.int64)
    wide = [m for m in multipliers(n) if int(np.float32(m)) != m]
    assert wide and max(wide) < 1 << 26 and Y_MAX * max(wide) + ((MAGIC_BITS + 1) << 32) < 1 << 63
    for m in wide + [1 << 25, 1 << 24, 1 << 23]:
        minus = (y < 0) if m & 0xFFF == 0 else 0
        bits = (y * m + (MAGIC_BITS << 32) + (1 << 31) - minus) >> 32
        assert np.array_equal(bits - MAGIC_BITS, np.sign(y) * ((np.abs(y) * m + (1 << 31)) >> 32)), m


def test_library_float_form_of_every_multiplier(tmp_path):
    ms = sorted(set().union(*map(multipliers, NS)))
    src = tmp_path / "rule.cu"
    src.write_text('#include <cstdio>\n#include "kernels.cuh"\nint main() { unsigned m; float v[2]; while (fread(&m, 4, 1, stdin)) '
                   '{ v[1] = dctgb::quant_multiplier(m, v[0]); fwrite(v, 4, 2, stdout); } }\n')
    exe = str(tmp_path / "rule")
    subprocess.run([build._nvcc()] + build.ARCH + ["-std=c++17", "-I" + build.INCLUDE, "-I" + build.CSRC, "-o", exe, str(src)],
                   check=True, capture_output=True)
    out = subprocess.run([exe], input=np.array(ms, dtype=np.uint32).tobytes(), check=True, capture_output=True).stdout
    for m, (f, fits) in zip(ms, np.frombuffer(out, dtype=np.float32).reshape(-1, 2)):
        assert (fits == 1) == (int(np.float32(m)) == m), m
        if fits:
            want = np.float32(m * 2.0 ** -32)
            assert f == (np.nextafter(want, np.float32(1)) if m & 0xFFF == 0 else want), m
