"""The lazy transforms of the compiled prime-power rings (primes of at most 50 bits)
and the canonical ones (wider primes) at the residues that drive their bounds:
every value q - 1, q - 1 alternating with 0, and random residues, all exact."""
import numpy as np
import pytest
import torch

import paper_2509_01253_gb300 as sf

pytestmark = pytest.mark.gpu

RINGS = [(3, 3), (3, 4), (3, 7), (5, 2), (5, 3), (5, 5), (7, 2), (7, 4)]


def _digit_rev(j, t, alpha):
    r = 0
    for _ in range(alpha):
        r, j = r * t + j % t, j // t
    return r


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("bits", [24, 50, 51, 61])
@pytest.mark.parametrize("t,alpha", RINGS)
def test_pp_transforms_at_extreme_residues(t, alpha, bits):
    L = 2
    r = sf.sf_pp_ring_create(t, alpha, L, bits, 0)
    try:
        info = sf.sf_pp_ring_info(r, L)
        M, mods = info["M"], info["moduli"]
        rng = np.random.default_rng(M + bits)
        a = np.zeros((4, L, M), dtype=np.uint64)
        for i, q in enumerate(mods):
            a[0, i] = q - 1
            a[1, i, ::2] = q - 1
            a[2, i, 1::2] = q - 1
            a[3, i] = rng.integers(0, q, M, dtype=np.uint64)
        A = _dev(np.zeros_like(a))
        sf.sf_pp_ntt(r, _dev(a), A, 4, False)
        ha = _host(A)
        x = np.zeros((1, L, M), dtype=np.uint64)
        x[0, :, 1] = 1
        X = _dev(x)
        sf.sf_pp_ntt(r, X, X, 1, False)
        hx = _host(X)[0]
        # residues of the inverse transform's inputs at their bound as well
        B = _dev(a)
        sf.sf_pp_ntt(r, B, B, 4, True)
        hb = _host(B)
        for i, q in enumerate(mods):
            assert (ha[:, i] < q).all() and (hb[:, i] < q).all()
            w = int(hx[i, _digit_rev(1, t, alpha)])
            assert pow(w, M, q) == 1 and pow(w, M // t, q) != 1
            for p in range(4):
                for j in [0, 1, M - 1, *rng.choice(M, 4, replace=False).tolist()]:
                    wk, want, back = pow(w, _digit_rev(int(j), t, alpha), q), 0, 0
                    for c in reversed(a[p, i].tolist()):
                        want = (want * wk + c) % q
                    assert int(ha[p, i, j]) == want, (p, i, j)
                    # coefficient j of the inverse: M^-1 sum_k a[rev(k)] omega^(-j k)
                    wj = pow(w, -int(j), q)
                    for k in reversed(range(M)):
                        back = (back * wj + int(a[p, i, _digit_rev(k, t, alpha)])) % q
                    assert int(hb[p, i, j]) == back * pow(M, -1, q) % q, (p, i, j)
        sf.sf_pp_ntt(r, A, A, 4, True)
        assert (_host(A) == a).all()
    finally:
        sf.sf_pp_ring_destroy(r)
