"""The batch solver's flat (request, prime) index space at its edges: tiles of
2,048 indices that end at, just before and just after a request, tiles that
span hundreds of requests, requests without primes, and every kind's repeated
primes.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# pi(17,863) = 2,048, the limit being 2n for kinds 0 and 1 and n for kind 2
BATCHES = {
    "tile_exact": [(2, 17863)],
    "tile_less_one": [(2, 17851), (0, 9)],
    "tile_plus_one": [(2, 17881), (1, 50)],
    "tiles_and_empty": [(0, 0), (2, 17863), (2, 1), (0, 8932), (1, 0), (1, 8931), (2, 0)],
    "many_small": [(k % 3, k % 97) for k in range(1500)],
    "small_then_large": [(k % 3, 1 + k % 5) for k in range(700)] + [(0, 60000), (2, 5000)],
    "only_empty": [(0, 0), (1, 0), (2, 1)],
}


@pytest.mark.parametrize("name", sorted(BATCHES))
def test_flat_index_edges(ctx, cat_lib, orc, name):
    reqs = BATCHES[name]
    out, offs, lens = cat_lib.cat_exact_batch(ctx, reqs)
    h = out.detach().cpu().numpy().view(np.uint32)
    want = {}
    for (kind, n), o, k in zip(reqs, offs, lens):
        if (kind, n) not in want:
            want[kind, n] = orc.exact(kind, n)
        got = h[int(o):int(o) + int(k)]
        w = want[kind, n]
        assert got.shape == w.shape and (got == w).all(), (kind, n)
