"""The fused prime-power key switch against the exact oracle, residue by
residue: compiled and generic transforms, one to four limbs, primes up to 61
bits, negative automorphism indices, several ciphertexts per launch, residues
at the top of their range, and the index check before anything is written."""
import numpy as np
import pytest
import torch

import paper_2509_01253_gb300 as sf
from oracle import primepower as pp

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


def _rand(rng, mods, shape, n):
    out = np.zeros((*shape, len(mods), n), dtype=np.uint64)
    for j, q in enumerate(mods):
        out[..., j, :] = rng.integers(0, q, (*shape, n), dtype=np.uint64)
    return out


@pytest.mark.parametrize("t,alpha,L,bits,count,h", [
    (3, 3, 1, 50, 1, 2), (3, 5, 2, 50, 5, 4), (7, 3, 1, 40, 2, -8), (5, 3, 4, 50, 3, 6), (3, 4, 2, 61, 4, 10),
    (7, 2, 3, 61, 1, -5)])
def test_pp_keyswitch_fused_matches_oracle(t, alpha, L, bits, count, h):
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    r = sf.sf_pp_ring_create(t, alpha, L, bits, 0)
    try:
        info = sf.sf_pp_ring_info(r, L)
        N, M, mods = info["N"], info["M"], info["moduli"]
        E = pp.RnsRlwe(pp.Ring(t, alpha), mods)
        rng = np.random.default_rng(31 * t + alpha + L)
        ka, kb = _rand(rng, mods, (L,), N), _rand(rng, mods, (L,), N)
        ct = _rand(rng, mods, (count, 2), N)
        for j, q in enumerate(mods):
            ct[0, :, j, :3] = q - 1
            ka[0, j, :3] = q - 1
        d_ct, d_ka, d_kb = _dev(ct), _dev(ka), _dev(kb)
        out = torch.full_like(d_ct, -1)
        with pytest.raises(sf.SafhireError):
            sf.sf_pp_keyswitch(r, d_ct, out, count, 2 * t, d_ka, d_kb)
        torch.cuda.synchronize()
        assert (out == -1).all()
        sf.sf_pp_keyswitch(r, d_ct, out, count, h, d_ka, d_kb)
        torch.cuda.synchronize()
        got = out.cpu().numpy().view(np.uint64)
        lists = lambda x: [[[int(v) for v in x[i, j]] for j in range(L)] for i in range(L)]
        for c in range(count):
            want = E.keyswitch(([[int(v) for v in ct[c, 0, j]] for j in range(L)],
                                [[int(v) for v in ct[c, 1, j]] for j in range(L)]), h % M, lists(ka), lists(kb))
            for part in range(2):
                for j in range(L):
                    assert got[c, part, j].tolist() == want[part][j], (c, part, j)
    finally:
        sf.sf_pp_ring_destroy(r)
