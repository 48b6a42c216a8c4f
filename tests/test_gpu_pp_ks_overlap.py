"""sf_pp_keyswitch between buffers that share words, the output a ciphertext (or
half of one) before or after the input: the words of the same call between
separate buffers.  The same buffer is refused, as by the header."""
import numpy as np
import pytest
import torch

import paper_2509_01253_gb300 as sf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,alpha,bits", [(5, 3, 50), (3, 7, 50), (3, 5, 55)])
def test_shifted_output(t, alpha, bits):
    L, count = 3, 40
    r = sf.sf_pp_ring_create(t, alpha, L, bits, 0)
    try:
        info = sf.sf_pp_ring_info(r, L)
        N, q = info["N"], info["moduli"]
        rng = np.random.default_rng(bits + alpha)
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()
        res = lambda *shape: dev(np.stack([rng.integers(0, m, (*shape, N), dtype=np.uint64) for m in q], axis=len(shape)))
        ka, kb, x = res(L), res(L), res(count, 2)
        want = torch.empty_like(x)
        sf.sf_pp_keyswitch(r, x, want, count, 1 + t, ka, kb)
        ct = 2 * L * N
        for shift in (-ct, ct, -ct // 2, ct // 2):
            buf = torch.zeros((count + 2) * ct, dtype=torch.int64, device="cuda")
            buf[ct:ct + count * ct] = x.flatten()
            out = buf[ct + shift:ct + shift + count * ct]
            sf.sf_pp_keyswitch(r, buf[ct:], out, count, 1 + t, ka, kb)
            torch.cuda.synchronize()
            assert torch.equal(out, want.flatten()), shift
        with pytest.raises(sf.SafhireError) as e:
            sf.sf_pp_keyswitch(r, x, x, count, 1 + t, ka, kb)
        assert e.value.status == sf.SF_EINVAL
    finally:
        sf.sf_pp_ring_destroy(r)
