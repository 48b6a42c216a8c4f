"""Key switches with digits of one to four limbs in launches that fill the GPU, where
the column kernels split neither the moduli nor the data limbs, and walk several
units a block: every ciphertext equals the same rotation in a launch of its own
(which splits them; compared with the oracle in test_gpu_passes), the product for
primes 2^50 - delta and Shoup's, up to N = 2^16."""
import numpy as np
import pytest

import paper_2509_01253_gb300 as sf
from _gpu import Session, dev_zeros, from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,L,bits,K,count", [
    (10, 7, 50, 4, 700), (10, 5, 50, 3, 700), (12, 8, 50, 4, 200), (13, 6, 45, 3, 100), (14, 4, 50, 2, 120),
    (14, 7, 45, 4, 60), (15, 5, 50, 3, 40), (16, 5, 50, 2, 24), (16, 6, 45, 4, 24), (16, 3, 50, 1, 40)])
def test_full_launches_equal_single_ones(log_n, L, bits, K, count):
    n, d = 1 << log_n, 2 * (1 << log_n) - 1
    s = Session(log_n, L, bits, K, sk_seed=41, rk_seed=42, rot_d=[d])
    try:
        rng = np.random.default_rng(43 + log_n + K)
        x = to_dev(np.stack([rng.integers(0, q, (count, 2, n), dtype=np.uint64) for q in s.info["moduli"][:L]], axis=2))
        got, one = dev_zeros(count, 2, L, n), dev_zeros(2, L, n)
        sf.sf_rotate(s.ctx, s.rk, d, x, got, count)
        for c in sorted({0, 1, count // 2, count - 2, count - 1, *rng.integers(0, count, 4).tolist()}):
            sf.sf_rotate(s.ctx, s.rk, d, x[c], one, 1)
            assert (from_dev(got[c]) == from_dev(one)).all(), c
        sf.sf_sync(s.ctx)
    finally:
        s.close()
