"""Phase 1 at the edges of its segments and counting units: the binomial kinds'
path (one read-back, one block for the seeds) against the same quantity as a
factorial ratio (Legendre's formula for every prime, radix grouping), on both
sides of every unit edge and of every change of the segment length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def same(a, b):
    import torch
    assert np.array_equal(a.exps, b.exps) and np.array_equal(a.offsets, b.offsets)
    assert a.primes_sieved == b.primes_sieved
    assert torch.equal(a.primes(), b.primes())


def check(cat_lib, ctx, n):
    f = cat_lib.catalan_factor(ctx, n, cat_lib.CAT_CENTRAL_BINOMIAL)
    g = cat_lib.cat_ratio_factor(ctx, [2 * n], [n, n])
    same(f, g)
    f.free()
    g.free()
    f = cat_lib.catalan_factor(ctx, n, cat_lib.CAT_CATALAN)
    g = cat_lib.cat_ratio_factor(ctx, [2 * n], [n, n + 1])
    same(f, g)
    f.free()
    g.free()


@pytest.mark.parametrize("n", [2, 3, 4, 31, 32, 33, 255, 8191, 8192, 8193, 16384, 65535, 65536,
                               65537, 100_000, 1_000_003])
def test_units(cat_lib, ctx, n):
    check(cat_lib, ctx, n)


@pytest.mark.parametrize("seg_log", [13, 14, 15, 16, 17])
@pytest.mark.parametrize("off", [0, 1])
def test_segment_length_changes(cat_lib, ctx, seg_log, off):
    # 2^seg_log odd numbers per segment up to 8 segments per SM, twice as many above
    check(cat_lib, ctx, ((8 * sms()) << seg_log) + off)
