"""The schoolbook levels by rows and Phase 1's segments against the CPU oracle
(their other tests compare two paths of the library, which could share an
error): tree products of enough 16-, 32- and 64-limb operands for the rows,
modulo two 62-bit primes, and factorisations on both sides of unit and segment
edges, group by group."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("kind", ["ones", "sparse", "random"])
@pytest.mark.parametrize("slot", [16, 32, 64])
def test_rows(cat_lib, orc, slot, kind):
    count = 2 * slot * 64 * sms() + 33  # two products per lane and SM
    rng = np.random.default_rng(slot)
    if kind == "ones":
        v = np.full(count, 0xFFFFFFFF, dtype=np.uint32)
    elif kind == "sparse":
        v = (np.uint32(1) << rng.integers(0, 32, count).astype(np.uint32)).astype(np.uint32)
    else:
        v = rng.integers(1, 1 << 32, count, dtype=np.uint64).astype(np.uint32)
    c = cat_lib.Context(0)
    try:
        c.set_profiling(True)
        got = cat_lib.product_tree(c, v).cpu().numpy().view(np.uint32)
        # 16 limbs always, 32 and 64 from here on
        assert c.profile()["comba_rows"][0] >= {16: 1, 32: 2, 64: 3}[slot]
    finally:
        c.close()
    for q in orc.check_primes(seed=slot, count=2, lower=1 << 61, bits=62):
        want = 1
        for x in v.tolist():
            want = want * x % q
        assert orc.limbs_mod(got, q) == want


def check(cat_lib, ctx, orc, kind, n):
    exps, offs, primes = orc.factor(kind, n)
    f = cat_lib.catalan_factor(ctx, n, kind)
    try:
        assert np.array_equal(f.exps, exps) and np.array_equal(f.offsets, offs)
        assert np.array_equal(f.primes().cpu().numpy().view(np.uint32), primes)
        assert f.primes_sieved == orc.prime_count(orc.prime_limit(kind, n))
    finally:
        f.free()


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("n", [2, 3, 33, 8191, 8192, 8193, 16384, 65536, 100_000, 1_000_003])
def test_units(cat_lib, ctx, orc, kind, n):
    check(cat_lib, ctx, orc, kind, n)


@pytest.mark.parametrize("seg_log", [13, 14, 15])
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("kind", [0, 1])
def test_segment_length_changes(cat_lib, ctx, orc, kind, seg_log, off):
    # 2^seg_log odd numbers per segment up to 8 segments per SM, twice as many above
    check(cat_lib, ctx, orc, kind, ((8 * sms()) << seg_log) + off)
