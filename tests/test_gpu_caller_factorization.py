"""cat_reconstruct of a caller's own factorisation with more groups than the
library's binomial kinds have (the bit-decomposed form): given by the primes on
the device and the host arrays alone, with groups that start past the first
prime, empty groups, exponents of 0 and of 2^32 and more."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def reconstruct(cat_lib, ctx, primes, exps, offsets, cap):
    import torch
    d = torch.from_numpy(np.asarray(primes, dtype=np.uint32).view(np.int32)).cuda()
    e = (ctypes.c_uint64 * len(exps))(*exps)
    o = (ctypes.c_uint64 * len(offsets))(*offsets)
    f = cat_lib.Factorization(num_groups=len(exps), num_primes=len(primes),
                              primes_sieved=len(primes), exps=None, offsets=None,
                              primes=d.data_ptr(), host_exps=e, host_offsets=o)
    out = torch.zeros(cap, dtype=torch.int32, device="cuda")
    n = ctypes.c_size_t()
    ctx.check(cat_lib.load().cat_reconstruct(ctx.handle, ctypes.byref(f), cat_lib._ptr(out), cap,
                                             ctypes.byref(n), cat_lib._stream(None)))
    return out[:n.value]


def as_int(t):
    return int.from_bytes(t.cpu().numpy().view("<u4").tobytes(), "little")


def value(primes, exps, offsets):
    v = 1
    for g, e in enumerate(exps):
        for p in primes[offsets[g]:offsets[g + 1]]:
            v *= int(p) ** e
    return v


def groups(orc, count, per):
    """`count` groups of `per` primes each (group 3 empty), exponents 1, 2, .."""
    primes = orc.sieve(100_000)[:count * per]
    offsets = [min(g, 3) * per + max(0, g - 4) * per for g in range(count + 1)]
    return primes[:offsets[-1]], [g + 1 for g in range(count)], offsets


@pytest.mark.parametrize("count,per", [(65, 1), (70, 3), (300, 2)])
def test_host_arrays_alone(ctx, cat_lib, orc, count, per):
    primes, exps, offsets = groups(orc, count, per)
    want = value(primes, exps, offsets)
    got = reconstruct(cat_lib, ctx, primes, exps, offsets, want.bit_length() // 32 + 1)
    assert as_int(got) == want


def test_groups_past_the_first_prime(ctx, cat_lib, orc):
    primes, exps, offsets = groups(orc, 70, 2)
    shifted = np.concatenate([np.array([101, 103, 107], dtype=np.uint32), primes])
    want = value(primes, exps, offsets)
    got = reconstruct(cat_lib, ctx, shifted, exps, [o + 3 for o in offsets],
                      want.bit_length() // 32 + 1)
    assert as_int(got) == want


def test_exponents_of_zero(ctx, cat_lib, orc):
    primes, exps, offsets = groups(orc, 70, 1)
    assert as_int(reconstruct(cat_lib, ctx, primes, [0] * 70, offsets, 4)) == 1
    exps = [e if e % 3 else 0 for e in exps]
    want = value(primes, exps, offsets)
    got = reconstruct(cat_lib, ctx, primes, exps, offsets, want.bit_length() // 32 + 1)
    assert as_int(got) == want


@pytest.mark.parametrize("e", [1 << 32, (1 << 40) + 5, (1 << 64) - 1])
def test_long_exponents_of_one(ctx, cat_lib, orc, e):
    primes, exps, offsets = groups(orc, 66, 1)
    want = value(primes, exps, offsets)
    got = reconstruct(cat_lib, ctx, np.append(primes, np.uint32(1)), exps + [e],
                      offsets + [offsets[-1] + 1], want.bit_length() // 32 + 1)
    assert as_int(got) == want


def test_power_of_two_past_32_bits(ctx, cat_lib, orc):
    """2^(2^32 + 1) times a short number."""
    primes, exps, offsets = groups(orc, 66, 1)
    odd = value(primes, exps, offsets)
    zeros, e = 1 << 27, (1 << 32) + 1
    got = reconstruct(cat_lib, ctx, np.append(primes, np.uint32(2)), exps + [e],
                      offsets + [offsets[-1] + 1], zeros + odd.bit_length() // 32 + 2)
    assert not got[:zeros].any().item()
    assert as_int(got[zeros:]) == 2 * odd
