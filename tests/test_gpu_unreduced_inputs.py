"""sf_pack, sf_pack_gamma and sf_rotate_noalloc do not check their inputs'
residues: residues that are not below their modulus (up to 4q here, the
transforms' input range) give the outputs of their canonical representatives."""
import numpy as np
import pytest

import paper_2509_01253_gb300 as sf
from _gpu import Session, dev_zeros, from_dev, to_dev

pytestmark = pytest.mark.gpu


def residues(rng, shape, moduli, n):
    """(canonical, the same plus 0 .. 3 times the modulus)"""
    c = np.stack([rng.integers(0, q, (*shape, n), dtype=np.uint64) for q in moduli], axis=len(shape))
    k = rng.integers(0, 4, c.shape, dtype=np.uint64)
    return c, c + k * np.array(moduli, dtype=np.uint64)[:, None]


# 50 bits: the product for primes 2^50 - delta; 45 and 30: Shoup's; one- and two-limb digits
@pytest.mark.parametrize("log_n,L,bits,K", [(10, 3, 50, 1), (11, 3, 50, 2), (11, 3, 45, 1), (12, 2, 30, 1)])
def test_unreduced_residues_stand_for_their_class(log_n, L, bits, K):
    s = Session(log_n, L, bits, K, sk_seed=95, rk_seed=96)
    try:
        n = 1 << log_n
        c, u = residues(np.random.default_rng(97 + bits), (5, 2), s.info["moduli"][:L], n)
        c, u = to_dev(c), to_dev(u)
        for gamma in (0, 2):
            want, got = dev_zeros(2, L, n), dev_zeros(2, L, n)
            for m in (5, 1):   # a padded tree, and the trace alone
                sf.sf_pack_gamma(s.ctx, s.rk, c, m, 8 if m > 1 else 1, gamma, want)
                sf.sf_pack_gamma(s.ctx, s.rk, u, m, 8 if m > 1 else 1, gamma, got)
                assert (from_dev(got) == from_dev(want)).all(), (gamma, m)
        want, got = dev_zeros(2, 2, L, n), dev_zeros(2, 2, L, n)
        for d in (3, n + 1):
            sf.sf_rotate(s.ctx, s.rk, d, c, want, 2)
            sf.sf_rotate_noalloc(s.ctx, s.rk, d, u, got, 2)
            assert (from_dev(got) == from_dev(want)).all(), d
        sf.sf_sync(s.ctx)
    finally:
        s.close()
