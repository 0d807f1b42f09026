"""Index rules of the prefilter (csrc/row_runs.h), compiled for the host. Unaligned rows are read as
aligned 4-byte words: the rule that keeps them inside the caller's buffer, against the bytes each
run would read. The whole-sample mirror, against Python's integers, up to the longest side."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_12941_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("row_runs")
    src, so = str(d / "runs.cpp"), str(d / "runs.so")
    with open(src, "w") as f:
        f.write('#include "row_runs.h"\n'
                'extern "C" int words_inside(int xa, int y, int W, int H, int b, unsigned s) {\n'
                '  return dic::words_inside(xa, y, W, H, b, s);\n}\n'
                'extern "C" int mirror(int near, int k, int n) {\n'
                '  return near ? dic::mirror_k<true>(k, n) : dic::mirror_k<false>(k, n);\n}\n')
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, src, "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("bytes_", [1, 2, 4])
def test_shifted_words_stay_inside_the_buffer(lib, bytes_):
    H, refused, outside = 5, 0, 0
    for W in range(192, 292):
        for base in range(0, 4, min(bytes_, 4)):                # the first pixel's byte within its word
            for stride in (W * bytes_, W * bytes_ + bytes_):
                end = base + (H - 1) * stride + W * bytes_      # one behind the last pixel's last byte
                for x0 in range(0, W, 32):
                    xa = x0 - 16
                    if xa < 0 or xa + 64 > W:                   # goes through the mirror
                        continue
                    for y in range(H):
                        first = base + y * stride + xa * bytes_
                        shift = first & 3
                        last = first - shift + 4 * (16 * bytes_ + (shift > 0))
                        assert first - shift >= 0
                        ok = lib.words_inside(xa, y, W, H, bytes_, shift)
                        assert not ok or last <= end, (W, base, stride, xa, y)
                        refused += not ok
                        outside += last > end
    # the rule refuses just the runs that would leave the buffer; FP32 rows need none
    assert refused == outside and (outside > 0) == (bytes_ < 4)


@pytest.mark.parametrize("n", [2, 3, 8, 9, 31, 191, 192, 193, 4096, 2 ** 30, 2 ** 30 + 1, 2 ** 30 + 2, 3 * 2 ** 29, 2 ** 31 - 200])
def test_mirror_up_to_the_longest_side(lib, n):
    # a halo of 28 rows, or a run of 64 from 16 before the image or up to 80 behind its last column
    for k in list(range(-40, 64)) + list(range(n - 70, n + 150)):
        m = abs(k) % (2 * (n - 1))
        assert lib.mirror(0, k, n) == min(m, 2 * (n - 1) - m), k
        if 192 <= n <= 2 ** 30:
            assert lib.mirror(1, k, n) == min(m, 2 * (n - 1) - m), k
