"""A request that fails for want of memory after Phase 1, on a stream that does
not wait for the null stream: everything is given back, in the stream's order,
and the context's next requests are exact."""
import pytest

from paper_2601_11621_gb300 import capi

pytestmark = pytest.mark.gpu


def test_factorial_of_a_batch_past_its_budget(orc, cat_lib):
    import torch
    s = torch.cuda.Stream()
    # the budget holds Phase 1 of 300,000! and not its tree
    c = capi.Context(0, hbm_budget_bytes=2 << 20)
    try:
        for _ in range(20):
            with pytest.raises(capi.CatError) as e:
                capi.cat_exact_batch(c, [(capi.CAT_FACTORIAL, 300_000)], stream=s)
            assert e.value.code == capi.CAT_ENOMEM
            assert c.memory()[0] == 0
            got = capi.to_numpy(capi.catalan_exact(c, 3000, stream=s))
            assert (got == orc.catalan(3000)).all()
    finally:
        c.close()
