"""The short division by 7 of the quantizers (a product with the rounded reciprocal and one correction by the exact remainder,
csrc/common.cuh) equals the division, over all fp32 mantissas of two exponents and a sample of every other. The same
sequence in C with the C library's fused multiply-add; the GPU tests compare scales bit for bit besides."""
import ctypes
import subprocess

SOURCE = r"""
#include <math.h>
#include <stdint.h>
#include <string.h>
// mismatches among the floats of the patterns first, first + step, .. below last
extern "C" long long div7_mismatches(uint32_t first, uint32_t last, uint32_t step) {
  const float y = 1.0f / 7.0f;
  long long bad = 0;
  for (uint64_t b = first; b < last; b += step) {
    const uint32_t p = (uint32_t)b;
    float x;
    memcpy(&x, &p, 4);
    const float q = x * y;
    const float r = fmaf(fmaf(-7.0f, q, x), y, q), want = x / 7.0f;
    bad += memcmp(&r, &want, 4) != 0;
  }
  return bad;
}
"""


def test_short_division_by_seven(tmp_path):
    src, lib = tmp_path / "div7.cpp", tmp_path / "div7.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-O2", "-mfma", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(lib), str(src)])
    f = ctypes.CDLL(str(lib)).div7_mismatches
    f.restype, f.argtypes = ctypes.c_longlong, [ctypes.c_uint32] * 3
    for e in (127, 254):
        assert f(e << 23, (e + 1) << 23, 1) == 0, e
    assert f(0, 28 << 23, 331) == 0        # subnormals among the operands or the remainders: slow to compute with
    assert f(28 << 23, 255 << 23, 97) == 0
