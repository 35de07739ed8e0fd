"""The transform's 64-bit coefficients at the edges of its paths (through the
C ABI, bit-exact): the largest coefficients every prime set must hold, and
operands of odd lengths and odd alignment on both sides of each path's limit
(one block up to 4,096 product limbs, a row pass alone up to 8,192, column
passes above)."""
import numpy as np
import pytest

from paper_2601_11621_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def host(t):
    return t.detach().cpu().numpy().view(np.uint32)


# 2^22, 2^25 and 2^26 limbs fill the transforms of the three prime sets
@pytest.mark.parametrize("k", [2, 16, 2048, 4096, 8192, 1 << 22, 1 << 25, 1 << 26])
def test_largest_coefficients(ctx, cat_lib, k):
    """(2^(32 k) - 1)^2 = 2^(64 k) - 2^(32 k + 1) + 1 by two operands (not the
    squaring path): every coefficient is the largest of its position."""
    import torch
    a = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    got = cat_lib.bigint_mul(ctx, a, a.clone())
    want = torch.zeros(2 * k, dtype=torch.int32, device="cuda")
    want[0] = 1
    want[k] = -2
    want[k + 1:] = -1
    assert got.numel() == 2 * k and torch.equal(got, want)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("na,nb", [(1, 1), (1, 2), (3, 3), (33, 30), (2047, 2048), (4095, 1),
                                   (4096, 1), (4097, 3), (3001, 2999), (4097, 4095), (8191, 1),
                                   (1, 8191), (8192, 1), (5001, 3193), (9001, 9002)])
def test_odd_lengths_and_alignment(ctx, cat_lib, orc, na, nb, offset):
    """Operands of odd lengths (a last coefficient of one limb), starting
    `offset` limbs into their buffers, whose neighbouring words are not zero."""
    import torch
    a, b = W.random_limbs32(na, seed=na), W.random_limbs32(nb, seed=nb + 1)
    ta = torch.full((na + 8,), -1, dtype=torch.int32, device="cuda")
    tb = torch.full((nb + 8,), -1, dtype=torch.int32, device="cuda")
    ta[offset:offset + na] = torch.from_numpy(a.view(np.int32)).cuda()
    tb[offset:offset + nb] = torch.from_numpy(b.view(np.int32)).cuda()
    got = host(cat_lib.bigint_mul(ctx, ta[offset:offset + na], tb[offset:offset + nb]))
    assert np.array_equal(got, orc.mul(a, b))


@pytest.mark.parametrize("n", [4096, 2049, 4097 // 2, 3000, 3501])
def test_square_by_the_row_pass(ctx, cat_lib, orc, n):
    import torch
    a = W.random_limbs32(n, seed=n)
    t = torch.from_numpy(a.view(np.int32)).cuda()
    assert np.array_equal(host(cat_lib.bigint_mul(ctx, t, t)), orc.mul(a, a))


@pytest.mark.parametrize("slot", [8, 16, 64, 256, 1024, 2048])
@pytest.mark.parametrize("nprod", [2, 33, 136, 137, 273, 274, 513])
def test_levels_on_both_sides_of_the_cluster_rule(ctx, cat_lib, orc, slot, nprod):
    """Product trees whose level at `slot` limbs has nprod products: few go by
    clusters of blocks, many by one block each (the rule's limits are 512
    products, 273 of 1,024-limb and 136 of 2,048-limb operands on 152 SMs), and
    a block takes several short products, the last one fewer.  The tree's
    levels run from 8 limbs up, so every size between is covered too."""
    count = nprod * 2 * slot - 5
    if count > 150_000:
        count = 150_000 + nprod
    v = W.random_values(count, seed=slot + nprod)
    got = host(cat_lib.product_tree(ctx, v))
    q = orc.check_primes(seed=slot, count=1, lower=1 << 61, bits=62)[0]
    want = 1
    for x in v.tolist():
        want = want * x % q
    assert orc.limbs_mod(got, q) == want


@pytest.mark.parametrize("s", [1500, 700_000, 3 << 20])
def test_carry_through_many_tiles(ctx, cat_lib, s):
    """a (1 + 2^(32 s)) with a = 1 and then s limbs of ones from limb s: the sum
    at limb s overflows and its carry runs through the next s limbs, across
    the tiles (2,048 limbs) and, at the largest, across the 1,024 tiles that
    one block of the carry kernel resolves."""
    a = np.zeros(2 * s, dtype=np.uint32)
    a[0] = 1
    a[s:] = 0xFFFFFFFF
    b = np.zeros(s + 1, dtype=np.uint32)
    b[0] = b[s] = 1
    got = host(cat_lib.bigint_mul(ctx, a, b))
    v = int.from_bytes(a.astype("<u4").tobytes(), "little")
    assert int.from_bytes(got.astype("<u4").tobytes(), "little") == v + (v << (32 * s))
