"""The kernels' branch-free quotient q = a rb, q + (a - b q) rb with rb the correctly rounded 1 / b (Markstein 1990) is the
correctly rounded a / b for every a and b of 2^-60 .. 2^60, not only for those that are tried.

Both significands in [1, 2) (powers of two only shift the result: nothing under- or overflows in that range).  rb is off by at most
2^-25 and the first q by at most 2^-23, so |a - b q| < 2^-22: rounding it costs at most 2^-47, and multiplying it by rb instead of
1 / b at most another 2^-47.  The sum that is rounded last is therefore within 2^-46 of a / b, and its rounding can differ from that
of a / b only if some midpoint m of two neighbouring numbers lies that close to a / b.  With a and b as 24-bit integers and
M = 2^24 m or 2^25 m (odd, of 25 bits; the second for quotients below 1), 2^24 a - b M or 2^25 a - b M is then an integer n of at
most 5, and not 0, as b M has more bits than a 24-bit number has.  For a given b and n there are a few such M (a linear congruence),
so all the pairs (a, b) in question can be listed: here for |n| <= 8."""
import ctypes as C
import subprocess

import numpy as np
import pytest

SOURCE = r"""
#include <math.h>
#include <stdint.h>
/* the pairs of first <= b < end with |n| <= 8: their number; written to a and b where these are given; *wrong: how many of them
 * the three operations do not round like the division */
int64_t near_midpoints(uint32_t first, uint32_t end, uint32_t *out_a, uint32_t *out_b, int64_t *wrong) {
    int64_t found = 0;
    *wrong = 0;
    for (uint32_t b = first; b < end; ++b) {
        const int t = __builtin_ctz(b);
        const uint64_t odd = b >> t;
        uint64_t inv = odd;                                     /* odd * inv = 1 modulo 2^64 */
        for (int i = 0; i < 5; ++i) inv *= 2 - odd * inv;
        const float fb = (float)b, rb = 1.0f / fb;
        for (int below = 0; below < 2; ++below) {
            const int bits = 24 + below;
            const uint64_t step = 1ull << (bits - t);
            for (int64_t n = -8; n <= 8; ++n) {
                if (n == 0 || n % (1 << t)) continue;           /* b M = -n modulo 2^bits: n has all of b's factors of two */
                const int64_t n_odd = n / (1 << t);
                if (!(n_odd & 1)) continue;                     /* M is odd */
                for (uint64_t M = ((1ull << 24) & ~(step - 1)) + ((uint64_t)(-n_odd) * inv & (step - 1)); M < 1ull << 25; M += step) {
                    if (M <= 1ull << 24) continue;
                    const uint64_t a = (b * M + (uint64_t)n) >> bits;
                    if (a < 1u << 23 || a >= 1u << 24 || (a < b) != below) continue;
                    const float fa = (float)(uint32_t)a, q = fa * rb;
                    *wrong += fmaf(fmaf(-fb, q, fa), rb, q) != fa / fb;
                    if (out_a) { out_a[found] = (uint32_t)a; out_b[found] = b; }
                    ++found;
                }
            }
        }
    }
    return found;
}
"""


@pytest.fixture(scope="module")
def near(tmp_path_factory):
    d = tmp_path_factory.mktemp("near")
    (d / "near.c").write_text(SOURCE)
    fma = ["-mfma"] if " fma " in open("/proc/cpuinfo").read() else []          # else the C library's, which is slow
    subprocess.check_call(["gcc", "-O2", "-ffp-contract=off", "-fno-fast-math", *fma, "-shared", "-fPIC", "-o", str(d / "near.so"), str(d / "near.c"), "-lm"])
    lib = C.CDLL(str(d / "near.so"))
    lib.near_midpoints.argtypes = [C.c_uint32, C.c_uint32, C.c_void_p, C.c_void_p, C.POINTER(C.c_int64)]
    lib.near_midpoints.restype = C.c_int64
    return lib.near_midpoints


def _pairs(near, first, end):
    wrong = C.c_int64()
    n = near(first, end, None, None, C.byref(wrong))
    a, b = np.zeros(n, np.uint32), np.zeros(n, np.uint32)
    near(first, end, a.ctypes.data, b.ctypes.data, C.byref(wrong))
    return a, b


def test_the_listed_pairs_are_those_next_to_a_midpoint(near):
    # against trying every numerator of a few denominators
    for b in (1 << 23, (1 << 23) + 1, (1 << 23) + 24, 9699328, 11184811, 16777214, 16777215):
        a = np.arange(1 << 23, 1 << 24, dtype=np.int64)
        bits = np.where(a < b, 25, 24)
        down = (a << bits) // b
        want = set()
        for M in (down, down + 1):
            n = (a << bits) - b * M
            want |= set(a[(np.abs(n) <= 8) & (n != 0) & (M % 2 == 1) & (M > 1 << 24) & (M < 1 << 25)].tolist())
        assert set(_pairs(near, b, b + 1)[0].tolist()) == want, b


def test_every_quotient_next_to_a_midpoint_is_rounded_correctly(near):
    wrong, found = C.c_int64(), 0
    for first in range(1 << 23, 1 << 24, 1 << 21):
        found += near(first, first + (1 << 21), None, None, C.byref(wrong))
        assert wrong.value == 0, first
    assert found > 30_000_000


@pytest.mark.gpu
def test_the_kernels_quotient_rounds_them_correctly_too(near):
    import torch
    from paper_2410_23208_b200 import k2d
    for first in range(1 << 23, 1 << 24, 1 << 21):
        a, b = (torch.from_numpy(x.astype(np.float32)).cuda() for x in _pairs(near, first, first + (1 << 21)))
        for sa, sb in ((2.0 ** -83, 2.0 ** 36), (1.0, 1.0), (2.0 ** 36, 2.0 ** -83)):        # up to both ends of the range
            _, q, _ = k2d.eval_quotients(a * sa, b * sb)
            assert torch.equal(q, (a * sa) / (b * sb)), first
