"""Unbalanced products whose chunk products are summed as residues: lengths
around whole chunks (one limb over, one short, tails shorter and longer than
the short operand), odd lengths, both orders, and operands of all ones (the
largest coefficients and carries).  Bit-exact against the CPU oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def operand(n, ones, seed):
    if ones:
        return np.full(n, 0xFFFFFFFF, dtype=np.uint32)
    v = np.random.default_rng(seed).integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    v[-1] |= 1
    return v


SIZES = []
for ny in (4099, 6000, 8192, 12287):
    chunk = ((1 << 14 if ny <= 8192 else 1 << 15) - ny) & ~7
    for nx in (3 * chunk, 3 * chunk + 1, 4 * chunk - 1, 3 * chunk + ny // 2, 5 * chunk + ny + 3):
        SIZES.append((nx, ny))


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("ones", [False, True])
def test_chunked_sum_vs_oracle(ctx, cat_lib, orc, nx, ny, ones):
    x, y = operand(nx, ones, nx), operand(ny, ones, ny + 1)
    want = orc.mul(x, y)
    got = cat_lib.bigint_mul(ctx, x, y).cpu().numpy().view(np.uint32)
    assert got.shape == want.shape and (got == want).all()
    if not ones:
        got = cat_lib.bigint_mul(ctx, y, x).cpu().numpy().view(np.uint32)
        assert (got == want).all()


@pytest.mark.parametrize("k,ny", [(24, 5000001), (27, (1 << 26) - 5)])
def test_chunked_sum_of_long_transforms(ctx, cat_lib, k, ny):
    """The larger prime sets (2^23 and 2^26 points): operands of all ones, whose
    product is B^(nx+ny) - B^nx - B^ny + 1."""
    import torch
    nx = 2 * (((1 << k) - ny) & ~7) - 1
    x = torch.full((nx,), -1, dtype=torch.int32, device="cuda")
    got = cat_lib.bigint_mul(ctx, x, x[:ny])
    assert got.numel() == nx + ny
    want = torch.full_like(got, -1)
    want[:ny] = 0
    want[0] = 1
    want[nx] = -2
    assert torch.equal(got, want)


def test_chunked_sum_of_random_long_operands(ctx, cat_lib, orc):
    ny = 5000001
    nx = 2 * (((1 << 24) - ny) & ~7) - 1
    x, y = operand(nx, False, 1), operand(ny, False, 2)
    got = cat_lib.bigint_mul(ctx, x, y).cpu().numpy().view(np.uint32)
    for q in orc.check_primes(seed=5, count=2, lower=2 * 10**6, bits=62):
        want = int(orc.limbs_mod(x, q)) * int(orc.limbs_mod(y, q)) % q
        assert int(orc.limbs_mod(got, q)) == want


def test_chunked_sum_within_a_budget(cat_lib, orc):
    """Two chunks, the second short, in a budget with room for the first one's
    product but not for all residues at once (38 and 50 bytes per limb of a
    chunk's transform)."""
    L, ny = 1 << 17, 40000
    nx = ((L - ny) & ~7) + 5000
    x, y = operand(nx, False, 7), operand(ny, False, 8)
    tight = cat_lib.Context(0, hbm_budget_bytes=44 * L)
    want = orc.mul(x, y)
    tight.set_profiling(True)
    got = cat_lib.bigint_mul(tight, x, y).cpu().numpy().view(np.uint32)
    assert "overlap_tiles" in tight.profile()
    assert got.shape == want.shape and (got == want).all()
