"""The canonical transforms of M = 3^7 (primes of more than 50 bits) on either
side of the count from which they run in smaller blocks: the same words as the
transforms of a few polynomials at a time."""
import numpy as np
import pytest
import torch

import paper_2509_01253_gb300 as sf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("L,count", [(2, 304), (2, 305), (1, 608), (1, 609)])
def test_block_sizes_agree(L, count, inverse):
    r = sf.sf_pp_ring_create(3, 7, L, 55, 0)
    try:
        info = sf.sf_pp_ring_info(r, L)
        rng = np.random.default_rng(count)
        x = np.stack([rng.integers(0, q, (count, info["M"]), dtype=np.uint64) for q in info["moduli"]], axis=1)
        x = torch.from_numpy(x.view(np.int64)).cuda()
        y, few = torch.empty_like(x), torch.empty_like(x)
        sf.sf_pp_ntt(r, x, y, count, inverse)
        for c in range(0, count, 7):
            k = min(7, count - c)
            sf.sf_pp_ntt(r, x[c:], few[c:], k, inverse)
        torch.cuda.synchronize()
        assert torch.equal(y, few)
    finally:
        sf.sf_pp_ring_destroy(r)
