"""Where a budget decides between the two ways of an unbalanced product: one
block of scratch for all chunks' residues is taken when it fits to the byte,
and a budget one allocation unit shorter goes by chunks in turn.  Both exact,
with everything given back."""
import numpy as np
import pytest

from paper_2601_11621_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PRIMES, TILE = 5, 2048


def scratch_bytes(nx, ny, k):
    """Residues of n chunks of x, of y and of n products at 2^(k-1) points, and
    a byte per tile of the result, rounded up to the 256-byte unit."""
    m = ((1 << k) - ny) & ~7
    n = -(-nx // m)
    words = (2 * n + 1) * PRIMES * (1 << (k - 1)) + -(-(-(-(nx + ny) // TILE)) // 4)
    return -(-4 * words // 256) * 256


@pytest.mark.parametrize("short", [0, 256])
def test_room_is_taken_to_the_byte(cat_lib, orc, short):
    k, ny = 17, 40000
    nx = (((1 << k) - ny) & ~7) + 5000  # two chunks, the second short
    x, y = W.random_limbs32(nx, seed=1), W.random_limbs32(ny, seed=2)
    budget = scratch_bytes(nx, ny, k) - short
    c = cat_lib.Context(0, hbm_budget_bytes=budget)
    try:
        c.set_profiling(True)
        got = cat_lib.bigint_mul(c, x, y).cpu().numpy().view(np.uint32)
        assert ("overlap_tiles" in c.profile()) == (short > 0)
        in_use, peak = c.memory()
        assert in_use == 0 and (peak == budget if not short else peak < budget)
    finally:
        c.close()
    assert np.array_equal(got, orc.mul(x, y))
