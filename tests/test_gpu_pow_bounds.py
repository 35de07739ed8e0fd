"""bigint_pow where the length bound of its chain decides: bases whose power
lies just above a power of 2^32 (a top limb of 1 over a stretch of zeros), and
the value 1 with large exponents.  Lengths and top limbs are known, the rest is
checked modulo two 62-bit primes from the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def host(t):
    return t.detach().cpu().numpy().view(np.uint32)


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


@pytest.mark.parametrize("m,e", [(10, 3), (2001, 5), (1000003, 3), (3670019, 7), (3670033, 7),
                                 (19209373, 91)])
def test_power_just_above_a_power_of_the_word_base(ctx, cat_lib, orc, m, e):
    """a = the first 100 bits of ceil(2^(32 m / e)), zeros, and a low word: its
    power lies between 2^(32 m) and 2^(32 m) (1 + 2^-90)."""
    w, f = divmod(32 * m, e)
    bits = min(w, 100)
    a = (root_head(f, e, bits) << (w - bits)) | (0x9E3779B97F4A7C15 >> max(0, 64 - (w - bits)))
    limbs = np.frombuffer(a.to_bytes(4 * ((a.bit_length() + 31) // 32), "little"), dtype="<u4")
    got = host(cat_lib.bigint_pow(ctx, limbs.astype(np.uint32), e))
    assert got.size == m + 1 and got[-1] == 1
    for q in orc.check_primes(seed=m, count=2, lower=1 << 40, bits=62):
        assert orc.limbs_mod(got, q) == pow(int(orc.limbs_mod(limbs.astype(np.uint32), q)), e, q)


@pytest.mark.parametrize("e", [1, 2, (1 << 30) - 1, 1 << 40, (1 << 63) + 1])
def test_powers_of_one(cat_lib, e):
    """Into a buffer of one limb, in a budget that holds a few hundred limbs."""
    import ctypes

    import torch
    c = cat_lib.Context(0, hbm_budget_bytes=8 << 10)
    try:
        one = torch.ones(1, dtype=torch.int32, device="cuda")
        out = torch.zeros(1, dtype=torch.int32, device="cuda")
        n = ctypes.c_size_t()
        c.check(cat_lib.load().bigint_pow(c.handle, cat_lib._ptr(one), 1, e, cat_lib._ptr(out), 1,
                                          ctypes.byref(n), cat_lib._stream(None)))
        assert n.value == 1 and out.item() == 1
    finally:
        c.close()
