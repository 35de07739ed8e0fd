"""bigint_pow of bases whose buffers are zero above the value: the stretches
that the top scan walks down (1,024 limbs each) are whole, partly or not at all
zero, the first four of them (which one block scans) or more, and a base of
zeros alone is 0."""
import numpy as np
import pytest

from paper_2601_11621_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def power(cat_lib, ctx, limbs, pad, e):
    import torch
    a = torch.zeros(len(limbs) + pad, dtype=torch.int32, device="cuda")
    a[:len(limbs)] = torch.from_numpy(limbs.view(np.int32)).cuda()
    return cat_lib.bigint_pow(ctx, a, e).cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025])
@pytest.mark.parametrize("pad", [0, 1, 1022, 1023, 1024, 1025, 2048, 3071, 3072, 4095, 4096, 4097,
                                 50_000, 3_000_001])
def test_bases_with_zero_tops(ctx, cat_lib, orc, n, pad):
    a = W.random_limbs32(n, seed=n + 1)
    a[-1] |= 1
    assert np.array_equal(power(cat_lib, ctx, a, pad, 3), orc.power(a, 3))


@pytest.mark.parametrize("n", [1, 1024, 4096, 4097, 5000, 100_000])
def test_zero(ctx, cat_lib, n):
    assert power(cat_lib, ctx, np.zeros(n, dtype=np.uint32), 0, 2).size == 0


def test_one_block_scans_four_stretches_only(ctx, cat_lib):
    """Past them the whole chip scans: two launches (and their read-backs) more,
    whatever the zeros."""
    a = W.random_limbs32(1000, seed=5)
    a[-1] |= 1

    def launches(pad):
        power(cat_lib, ctx, a, pad, 3)
        before = cat_lib.load().cat_launch_count()
        power(cat_lib, ctx, a, pad, 3)
        return cat_lib.load().cat_launch_count() - before
    assert launches(4095) == launches(0)
    assert launches(4096) == launches(4_000_000) > launches(0)
