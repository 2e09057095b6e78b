"""soft64.h compiled for the host against the host's binary64 arithmetic: every
result it claims, over ordinary operands, ties, carries into the next binade
and borrows into the previous one, significands of few or all bits, and zeros,
subnormals, infinities and NaNs (which it must decline)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2604_27193_gb300", "csrc")

SRC = r"""
#include "soft64.h"
#include <stdio.h>
#include <stdlib.h>
#include <random>
using namespace aeb;
static double D(uint64_t b) { double x; memcpy(&x, &b, 8); return x; }
int main()
{
    std::mt19937_64 g(7);
    long muls = 0, adds = 0, wide = 0, wrong = 0, claimed_special = 0;
    for (long i = 0; i < 6000000; ++i) {
        const uint64_t r = g(), q = g(), t = g();
        const uint64_t F = 0xfffffffffffffull;
        int ea = 1023 + (int)(r % 81) - 40, eb = ea + 2 - (int)((r >> 8) % 68);
        if (i % 4 == 0) eb = ea - (int)((r >> 8) % 4);
        if (i % 32 == 0) { ea = (int)(r % 2048); eb = (int)((r >> 12) % 2048); }
        uint64_t ma = q & F, mb = t & F;
        if ((r >> 20) % 4 == 0) ma &= F << ((r >> 22) % 53);
        if ((r >> 30) % 4 == 0) mb &= F << ((r >> 32) % 53);
        if ((r >> 40) % 4 == 0) ma = F - (ma & 3);
        if ((r >> 42) % 4 == 0) ma &= 3;
        if ((r >> 44) % 8 == 0) mb = F - (mb & 7);
        ma &= F; mb &= F;
        const double a = D(((r >> 60) & 1) << 63 | (uint64_t)ea << 52 | ma);
        const double b = D(((r >> 61) & 1) << 63 | (uint64_t)eb << 52 | mb);
        if (soft_factor_ok(b)) {
            uint32_t bad = 0;
            const double p = soft_mul(a, soft_factor(b), bad), e = a * b;
            if (!soft_bad(bad)) {
                muls++;
                wrong += bits_of(p) != bits_of(e);
                claimed_special += ea == 0 || ea == 2047;
            }
        }
        if (ea < 23 || ea > 2023) continue;  // outside soft_add's stated range of a
        uint32_t n = 0, w = 0;
        const double s = soft_add<false>(a, b, n), u = soft_add<true>(a, b, w), e = a + b;
        if (!soft_bad(n)) { adds++; wrong += bits_of(s) != bits_of(e); }
        if (!soft_bad(w)) { wide++; wrong += bits_of(u) != bits_of(e); }
        claimed_special += (!soft_bad(n) || !soft_bad(w)) && (eb == 0 || eb == 2047);
    }
    printf("%ld %ld %ld %ld %ld\n", muls, adds, wide, wrong, claimed_special);
    return 0;
}
"""


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    d = tmp_path_factory.mktemp("soft64")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", f"-I{CSRC}", str(src), "-o",
                    str(exe)], check=True)
    return [int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True,
                                           text=True).stdout.split()]


def test_soft_arithmetic_is_the_hosts(counts):
    muls, adds, wide, wrong, special = counts
    assert wrong == 0 and special == 0
    # and it applies where the kernel uses it: nearly all products, the sums of
    # exponent differences it names
    assert muls > 5_000_000 and adds > 2_000_000 and wide > 4_000_000
