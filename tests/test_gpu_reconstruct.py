"""Reconstruction: groups with e >= 2 as repeated leaves of one tree or as
powers (the rule's two sides), and results written straight into the caller's
buffer or copied there."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def host(t):
    return t.detach().cpu().numpy().view(np.uint32)


def as_int(t):
    return int.from_bytes(host(t).astype("<u4").tobytes(), "little")


# (3n)! / n!^3: the primes in (n, 3n/2] have e = 2, about 4,096 leaves in all
# between n = 40,000 and n = 60,000 (more than that, and more than a quarter of
# the e = 1 primes, go by powers)
@pytest.mark.parametrize("n", [1, 2, 10, 100, 5_000, 20_000, 60_000, 100_000])
def test_repeated_groups(ctx, cat_lib, n):
    got = cat_lib.cat_ratio_exact(ctx, [3 * n], [n, n, n])
    assert as_int(got) == math.factorial(3 * n) // math.factorial(n) ** 3


@pytest.mark.parametrize("n", [1, 3, 500, 30_000, 100_003])
def test_result_buffers(ctx, cat_lib, n):
    """A buffer of exactly the result's length (below the bound: copied), of the
    bound's, longer and odd-aligned (written in place, words past the bound
    untouched), and one limb short (CAT_ERANGE)."""
    import torch
    want = math.comb(2 * n, n) // (n + 1)
    need = (want.bit_length() + 31) // 32
    bound = cat_lib.cat_bound_limbs(n, cat_lib.CAT_CATALAN)
    for size, start in ((need, 0), (bound, 0), (bound + 7, 0), (bound + 7, 1)):
        buf = torch.full((size + start,), -3, dtype=torch.int32, device="cuda")
        out = buf[start:]
        got = cat_lib.catalan_exact(ctx, n, out=out)
        assert got.numel() == need and as_int(got) == want
        assert (out[max(need, bound):] == -3).all() and (buf[:start] == -3).all()
    if need > 1:
        with pytest.raises(cat_lib.CatError) as e:
            cat_lib.catalan_exact(ctx, n, out=torch.empty(need - 1, dtype=torch.int32,
                                                          device="cuda"))
        assert e.value.code == cat_lib.CAT_ERANGE
