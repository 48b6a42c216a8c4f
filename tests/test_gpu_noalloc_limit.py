"""sf_rotate_noalloc at its documented limit: the largest accepted count, in place
(the call that uses most of the fixed array), equals sf_rotate, and one more is
refused by a message that names the limit."""
import pytest

import paper_2509_01253_gb300 as sf
from _gpu import Session, dev_zeros, from_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,L,K,ks_batch", [(14, 3, 1, 512), (12, 8, 4, 512), (13, 7, 3, 512), (15, 4, 2, 1), (15, 4, 2, 512)])
def test_largest_count(log_n, L, K, ks_batch):
    n, dnum, nm = 1 << log_n, -(-L // K), L + K
    limbs = L + max(L, 2 * K) + max(dnum * nm, 2 * L) + 2 * L
    words = lambda c: 2 * c * 2 * L * n + limbs * n * min(c, ks_batch)
    count = max(c for c in range(1, 64) if words(c) <= 4 << 20)
    s = Session(log_n, L, 50, K, sk_seed=51, rk_seed=52, rot_d=[3])
    try:
        sf.sf_ctx_set_option(s.ctx, "ks_batch", ks_batch)
        x = s.encrypt([k % 777 for k in range((count + 1) * n)], 53, count + 1)
        want = dev_zeros(count, 2, L, n)
        sf.sf_rotate(s.ctx, s.rk, 3, x, want, count)
        with pytest.raises(sf.SafhireError) as e:
            sf.sf_rotate_noalloc(s.ctx, s.rk, 3, x, x, count + 1)
        assert e.value.status == sf.SF_EINVAL and "documented limit" in e.value.message
        sf.sf_rotate_noalloc(s.ctx, s.rk, 3, x, x, count)
        sf.sf_sync(s.ctx)
        assert (from_dev(x[:count]) == from_dev(want)).all()
    finally:
        s.close()
