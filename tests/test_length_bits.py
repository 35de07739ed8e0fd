"""The length bound of a chain of products (csrc/length_bits.h, plain host
arithmetic, compiled here): never below the true length and at most one limb
above it, for powers just above and just below a power of 2^32 (the bases of
524,291 limbs and more are those whose bits a double rounds down), for the
value 1 with exponents up to 2^63, and for random bases."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include "length_bits.h"
#include <algorithm>
#include <stdio.h>
int main()
{
    unsigned long long n, top, e;
    while (scanf("%llu %llu %llu", &n, &top, &e) == 3) {
        const double b = cat::top_bits(n, top);
        double x = b;
        unsigned long long len = n;
        int bit = 63;
        while (!(e >> bit & 1)) bit--;
        while (bit-- > 0) {
            x = cat::product_bits(x, x);
            len = std::min<unsigned long long>(2 * len, cat::bits_limbs(x));
            if (e >> bit & 1) {
                x = cat::product_bits(x, b);
                len = std::min<unsigned long long>(len + n, cat::bits_limbs(x));
            }
        }
        printf("%llu\n", len);
    }
}
"""


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    d = tmp_path_factory.mktemp("bits")
    (d / "driver.cpp").write_text(DRIVER)
    exe = str(d / "driver")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2601_11621_gb300", "csrc"),
                    str(d / "driver.cpp"), "-o", exe], check=True)

    def run(cases):
        text = "".join(f"{n} {top} {e}\n" for n, top, e in cases)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True)
        return [int(x) for x in out.stdout.split()]
    return run


def root_head(f, e, bits=100):
    """ceil(2^(f/e + bits)) for 0 <= f < e."""
    lo, hi = 1 << bits, 1 << (bits + 1)
    while lo < hi:
        mid = (lo + hi) // 2
        if mid ** e >= 1 << (bits * e + f):
            hi = mid
        else:
            lo = mid + 1
    return lo


def base_of(head, shift):
    """Length and top two limbs of head 2^shift."""
    n = (head.bit_length() + shift + 31) // 32
    s = shift - 32 * (n - 2)
    return n, head << s if s >= 0 else head >> -s


def near(m, e, above):
    """A base whose e-th power is just above (or just below) 2^(32 m), and the
    power's length."""
    w, f = divmod(32 * m, e)
    head = root_head(f, e) - (0 if above else 1)
    return (*base_of(head, w - 100), e), m + 1 if above else m


# 32 m / e: bases of 524,289 to 4.2 million limbs for e = 7, and bases of
# 211,093 and 185,366 limbs
EDGES = [(3670019, 7), (3670033, 7), (7340047, 7), (14680075, 7), (29360117, 7),
         (19209373, 91), (34663426, 187), (1000003, 3), (2001, 5), (10, 3)]


def test_powers_next_to_a_power_of_the_word_base(bounds):
    cases, want = zip(*[near(m, e, above) for m, e in EDGES for above in (True, False)])
    assert max(c[0] for c in cases) > 4_000_000
    for c, got, length in zip(cases, bounds(cases), want):
        assert length <= got <= length + 1, (c, got, length)


def test_a_sweep_of_such_bases(bounds):
    rng = random.Random(11)
    picks = [(rng.randrange(e, 1 << 27), e) for e in (3, 5, 7, 11, 91, 187) for _ in range(100)]
    cases, want = zip(*[near(m, e, True) for m, e in picks if m >= 4 * e])
    for c, got, length in zip(cases, bounds(cases), want):
        assert length <= got <= length + 1, (c, got, length)


def test_powers_of_one_stay_one_limb(bounds):
    cases = [(1, 1 << 32, e) for e in (1, 2, 1 << 40, (1 << 55) - 1, 1 << 63, (1 << 64) - 1)]
    assert bounds(cases) == [1] * len(cases)


def test_powers_of_two(bounds):
    # 2^(e k) has e k // 32 + 1 limbs exactly
    cases, want = [], []
    for k in (1, 31, 32, 63, 64, 32 * 524_291, 12_345_677):
        for e in (1, 2, 3, 31, 32, 33, 64):
            n = k // 32 + 1
            top = (1 << (k % 32 + 32)) if n > 1 else (1 << k) << 32
            cases.append((n, top, e))
            want.append(e * k // 32 + 1)
    for c, got, length in zip(cases, bounds(cases), want):
        assert length <= got <= length + 1, (c, got, length)


def test_random_short_bases(bounds):
    rng = random.Random(3)
    cases, want = [], []
    for _ in range(300):
        a = rng.getrandbits(rng.randrange(1, 400)) | 1
        e = rng.randrange(1, 60)
        cases.append((*base_of(a, 0), e) if a >> 32 else (1, a << 32, e))
        want.append(((a ** e).bit_length() + 31) // 32)
    for c, got, length in zip(cases, bounds(cases), want):
        assert length <= got <= length + 1, (c, got, length)
