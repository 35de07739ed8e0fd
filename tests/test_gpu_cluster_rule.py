"""Tree levels of one-block transforms on both sides of the rule that gives few
products a cluster of blocks each (spread_primes in csrc/ntt.cu): at its limit,
one past it, and with a last block that is not full.  The kernel profile says
which side every level took, the product is checked modulo a 62-bit prime."""
import numpy as np
import pytest

from paper_2601_11621_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SLOTS = [128, 256, 512, 1024, 2048]  # schoolbook up to 64, multi-pass above 2048


def limit(slot):
    """The most products of slot-limb operands (slot points) by clusters: their
    five blocks of slot / 4 threads (at least a warp) about once around the
    chip, at most 512."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return min(512, sms * 2048 * 9 // (5 * 8 * max(32, slot // 4)))


def expected(count):
    """Launches of a tree over count 32-bit values (8 to a node): clusters, one block."""
    out = {"ntt_mul_cluster": 0, "ntt_mul_fused": 0}
    nodes, slot = -(-count // 8), 8
    while nodes > 1:
        if slot in SLOTS:
            few = nodes // 2 <= limit(slot)
            out["ntt_mul_cluster" if few else "ntt_mul_fused"] += 1
        nodes, slot = -(-nodes // 2), 2 * slot
    return out


@pytest.mark.parametrize("slot", SLOTS)
@pytest.mark.parametrize("past", [0, 1, 34])
def test_levels_around_the_limit(cat_lib, orc, slot, past):
    count = (limit(slot) + past) * 2 * slot - 5
    v = W.random_values(count, seed=slot + past)
    c = cat_lib.Context(0)
    try:
        assert c.tuning()[0] == 64  # the default crossover
        c.set_profiling(True)
        got = cat_lib.product_tree(c, v).cpu().numpy().view(np.uint32)
        ran = c.profile()
    finally:
        c.close()
    want = expected(count)
    assert want["ntt_mul_fused"] > 0 or slot == SLOTS[0] and not past
    assert {k: ran[k][0] if k in ran else 0 for k in want} == want
    q = orc.check_primes(seed=slot, count=1, lower=1 << 61, bits=62)[0]
    r = 1
    for x in v.tolist():
        r = r * x % q
    assert orc.limbs_mod(got, q) == r
