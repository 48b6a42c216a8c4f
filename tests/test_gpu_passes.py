"""The register-resident passes and the coefficient-domain key switch where
their forms change, bit for bit against the oracle: every digit width (K = 1 ..
4, ragged last digits), moduli that admit the 50-bit product and moduli that do
not, data and special primes of different sizes, residues at the top of their
range, launches that split the moduli and launches that fill the GPU, and a
round whose leaves sum over more input ciphertexts than one lazy sum holds."""
import numpy as np
import pytest

import paper_2509_01253_gb300 as sf
from paper_2509_01253_gb300 import workloads as wl
from _gpu import Session, dev_zeros, from_dev, gpu_layer, oracle_layer, oracle_params, stream_input, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,L,bits,K,special", [
    (10, 6, 50, 3, 50), (10, 7, 50, 4, 50), (11, 5, 50, 4, 50), (10, 8, 50, 1, 50), (13, 2, 50, 2, 50),
    (11, 3, 49, 1, 49), (10, 3, 33, 2, 50), (10, 3, 50, 1, 30), (10, 3, 20, 1, 20), (12, 2, 30, 1, 30)])
def test_rotate_every_digit_and_modulus_form(oracle, log_n, L, bits, K, special):
    n = 1 << log_n
    ds = [3, n // 2 + 1, n + 1, 2 * n - 1]
    s = Session(log_n, L, bits, K, special_bits=special, sk_seed=61, rk_seed=62, rot_d=ds)
    try:
        prm = oracle_params(oracle, log_n, L, bits, K, special)
        keys = oracle.rotation_keys(prm, oracle.keygen(prm, 61), 62, ds)
        q = s.info["moduli"][:L]
        rng = np.random.default_rng(7 + log_n + bits)
        cts = np.stack([np.stack([np.stack([rng.integers(0, m, n, dtype=np.uint64) for m in q]) for _ in range(2)])
                        for _ in range(2)])
        for i, m in enumerate(q):
            cts[1, :, i] = m - 1
        d_ct = to_dev(np.concatenate([cts, np.repeat(cts[:1], 9, axis=0)]))
        for d in ds:
            want = [oracle.rotate(prm, keys, d, cts[x]) for x in range(2)]
            for count in (1, 2, 11):
                out = dev_zeros(count, 2, L, n)
                sf.sf_rotate(s.ctx, s.rk, d, d_ct, out, count)
                got = from_dev(out)
                for x in range(count):
                    assert (got[x] == want[1 if x == 1 else 0]).all(), (d, count, x)
    finally:
        s.close()


def test_round_over_many_input_ciphertexts(oracle):
    """20 input ciphertexts at N = 2^10 (a lazy sum holds 16)."""
    log_n, L, K = 10, 2, 1
    case = wl.fc_case(71, 20 * 1024 - 5, 3)
    delta = 2.0 ** 20
    s = Session(log_n, L, 50, K, sk_seed=72, rk_seed=73)
    try:
        prm = oracle_params(oracle, log_n, L, 50, K)
        s_o = oracle.keygen(prm, 72)
        keys = oracle.rotation_keys(prm, s_o, 73)
        xs = stream_input(case)
        d_in = s.encrypt(sf.sf_encode_input(xs, delta), 74, 20)
        lay = gpu_layer(s, case, delta, delta ** 2)
        out = dev_zeros(1, 2, L, s.n)
        sf.sf_eval_linear_layer(s.ctx, lay, s.rk, d_in, 20, case.sigma_prev, case.sigma_out, out, 1)
        sf.sf_sync(s.ctx)
        cts = oracle.encrypt(prm, s_o, oracle.quantize(xs, delta), 74, 20)
        want = oracle.eval_linear_layer(prm, oracle_layer(oracle, case, delta, delta ** 2), keys, cts,
                                        case.sigma_prev, case.sigma_out)
        assert (from_dev(out) == want).all()
        sf.sf_layer_destroy(lay)
    finally:
        s.close()
