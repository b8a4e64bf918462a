"""The operand scratch of the tensor-core ciphertext-diagonal product holds every slice of every pass,
for all diagonal counts (no GPU: the sizes' header compiled by the host compiler)."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_00482_gb300", "csrc")
SRC = """
#include <string.h>

#include "he_cdiag_tc_plan.h"
// the loops of cdiag_tc_mac: bytes written by the largest slice of any pass
extern "C" int64_t used(int sms, int tiles, int mods, int n_ct) {
    int64_t most = 0;
    for (int i0 = 0; i0 < n_ct; i0 += TC_DIAGS) {
        const TcPass p = tc_pass(sms, mods, n_ct, i0);
        for (int first = 0; first < tiles; first += p.slice)
            most = std::max(most, std::min(p.slice, tiles - first) * p.tile_bytes);
    }
    return most;
}
extern "C" int64_t scratch(int sms, int tiles, int mods, int n_ct) { return tc_scratch_bytes(sms, tiles, mods, n_ct); }
extern "C" int32_t digit_sum(int n, const float *y, const int32_t *h) {
    uint32_t sum = 0;
    for (int m = 0; m < n; ++m) sum = tc_digit_init(sum, h[m]);
    for (int m = 0; m < n; ++m) {
        const float f = y[m] + 12582912.0f;  // 1.5 2^23
        uint32_t bits;
        memcpy(&bits, &f, 4);
        sum = tc_digit_add(sum, bits, h[m]);
    }
    return (int32_t)sum;
}
extern "C" int min_diags(const uint64_t *primes, int nl, int64_t n, int64_t k) { return tc_min_diags(primes, nl, n, k); }
extern "C" int moduli(uint64_t q) { return tc_moduli(q); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    so = str(d / "plan.bin")
    subprocess.run(["g++", "-std=c++20", "-O1", "-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error", "-shared", "-fPIC", "-I", CSRC, str(d / "plan.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for f in (lib.used, lib.scratch):
        f.restype, f.argtypes = ctypes.c_int64, [ctypes.c_int] * 4
    lib.moduli.argtypes = [ctypes.c_uint64]
    return lib


@pytest.mark.parametrize("tiles", [128, 256, 512, 768, 3584])
@pytest.mark.parametrize("sms", [132, 148, 152])
def test_scratch_holds_every_pass(lib, sms, tiles):
    for mods in range(1, 16):
        for n_ct in range(1, 1025):
            assert lib.used(sms, tiles, mods, n_ct) <= lib.scratch(sms, tiles, mods, n_ct), (mods, n_ct)


def test_a_short_last_pass_can_need_more_than_a_full_one(lib):
    """The N = 2^12 ring's and an all-40-bit chain's moduli, the diagonal counts that outgrew a scratch of the first pass's size."""
    mods = lib.moduli((1 << 40) - 87)
    assert mods == 10
    assert lib.scratch(152, 512, mods, 256) < lib.scratch(152, 512, mods, 300) == lib.used(152, 512, mods, 300)
    assert lib.scratch(152, 256, mods, 256) < lib.scratch(152, 256, mods, 449) == lib.used(152, 256, mods, 449)


def test_digit_sums_are_exact_without_signed_overflow(lib):
    """The largest terms and random ones; signed overflow would end the process (trapping sanitizer)."""
    lib.digit_sum.argtypes = [ctypes.c_int, ctypes.POINTER(ctypes.c_float), ctypes.POINTER(ctypes.c_int32)]
    rng = random.Random(1)
    for case in range(2000):
        n = rng.randint(1, 15)
        y = [rng.choice([-256, 255, rng.randint(-256, 256)]) for _ in range(n)]
        h = [rng.choice([-(1 << 19), 1 << 19, rng.randint(-(1 << 19), 1 << 19)]) for _ in range(n)]
        if case < 4:
            n, y, h = 15, [256 if case & 1 else -256] * 15, [(1 << 19) if case & 2 else -(1 << 19)] * 15
        want = sum(a * b for a, b in zip(y, h))
        assert abs(want) < 1 << 31
        assert lib.digit_sum(n, (ctypes.c_float * n)(*y), (ctypes.c_int32 * n)(*h)) == want


@pytest.mark.parametrize("bits,n,cols,want", [([40, 20], 64, 8, 11), ([40, 20], 2048, 128, 10), ([60, 40, 40], 32, 8, 18), ([60, 40, 40], 64, 8, 20),
                                              ([60, 40, 40], 4096, 8, 25), ([60] + [40] * 6, 16, 8, 14), ([60] + [40] * 6, 64, 8, 16),
                                              ([60] + [40] * 6, 256, 128, 15), ([60] + [40] * 6, 8192, 8, 20), ([60] + [40] * 6, 8192, 200, 12),
                                              ([60] + [40] * 6, 256, 30, 15), ([60] + [40] * 6, 256, 101, 12)])
def test_line_between_the_forms(lib, bits, n, cols, want):
    """tc_min_diags for the parameter sets' prime sizes (primes just below the powers of two)."""
    primes = (ctypes.c_uint64 * len(bits))(*[(1 << b) - 87 for b in bits])
    lib.min_diags.argtypes = [ctypes.POINTER(ctypes.c_uint64), ctypes.c_int, ctypes.c_int64, ctypes.c_int64]
    assert lib.min_diags(primes, len(bits), n, cols) == want
