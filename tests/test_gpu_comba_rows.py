"""The row-wise schoolbook levels of the product tree against the transforms:
the same product with the schoolbook crossover at 8 limbs (every level from 16
limbs up by transforms) and at 64.  Counts on both sides of two products per
lane and SM and counts that leave a warp's last lanes without a product;
values whose limbs are all ones, mostly zero, and random."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def contexts(cat_lib):
    out = []
    old = os.environ.get("CAT_COMBA_MAX_SLOT")
    try:
        for slot in ("8", "64"):
            os.environ["CAT_COMBA_MAX_SLOT"] = slot
            out.append(cat_lib.Context(0))
    finally:
        if old is None:
            del os.environ["CAT_COMBA_MAX_SLOT"]
        else:
            os.environ["CAT_COMBA_MAX_SLOT"] = old
    return out


def product(lib, ctx, v):
    d = torch.from_numpy(v.view(np.int32)).cuda()
    return lib.product_tree(ctx, d).cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("kind", ["ones", "sparse", "random"])
@pytest.mark.parametrize("extra", [-64, 0, 33, 4000])
@pytest.mark.parametrize("slot", [16, 32, 64])
def test_rows_equal_transforms(contexts, cat_lib, slot, extra, kind):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    count = 2 * slot * 64 * sms + extra
    rng = np.random.default_rng(1000 + slot + extra)
    if kind == "ones":
        v = np.full(count, 0xFFFFFFFF, dtype=np.uint32)
    elif kind == "sparse":
        v = (np.uint32(1) << rng.integers(0, 32, count).astype(np.uint32)).astype(np.uint32)
    else:
        v = rng.integers(1, 1 << 32, count, dtype=np.uint64).astype(np.uint32)
    want, got = (product(cat_lib, c, v) for c in contexts)
    assert got.shape == want.shape and (got == want).all()
