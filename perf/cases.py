"""Timing cases: the work that users of this library have it do, through its
public entry points.

Every output is whole numbers (residues modulo the ring's primes, or torus
words modulo 2^53).  The rings and layer shapes are those of
``paper_2509_01253_gb300.workloads`` (the four parameter sets and the
ResNet-20/-18/-34-shaped networks) and the paper's Table 2 (prime-power rings
and gadgets).

Case kinds:
  round      one linear-layer round (sf_eval_linear_layer, or the gamma = 2
             form that also reads the client's powers)
  batch      several uneven rounds in one call (sf_eval_layers), as the
             serving loop issues them
  rotate     automorphism + hybrid key switch of `count` ciphertexts
  ntt        batched negacyclic transform over every limb, either direction
  pp_ntt     length-M transform of a prime-power ring M = t^alpha
  pp_ks      RNS key switch after an automorphism in a prime-power ring
  tq_ks      torus (q = 2^53) gadget key switch of Table 2
"""
import functools
import math
import weakref

import numpy as np
import torch

import paper_2509_01253_gb300 as sf
from paper_2509_01253_gb300 import workloads as wl

TORUS = ((3, 7, 512, 3), (7, 4, 4096, 3), (7, 4, 65536, 2), (5, 5, 310, 5), (5, 5, 310, 4))


def listed():
    return [
        # The smallest round: a 64 x 64 fully connected layer at N = 2^12 with
        # 30-bit primes.  Few ciphertexts: launches and latency count.
        conv_round("fc64", "fc64", 1, 1, 64, 64, 1, 1, 0),
        # A single ciphertext rotated at the largest ring, as a client of the
        # building blocks calls it.
        {"name": "rotate_one_2e16", "kind": "rotate", "params": "r34", "count": 1, "d": 5},
        # ResNet-20, first stage: 3 x 3, 16 -> 16 channels on 32 x 32 at
        # N = 2^14; 16384 outputs in two packed ciphertexts.
        conv_round("resnet20_conv", "conv16", 32, 32, 16, 16, 3, 1, 1),
        # A later, strided ResNet-20 conv with the client's powers (gamma = 2):
        # half of the key switches, twice the leaf work.  8192 outputs.
        conv_round("resnet20_down_gamma2", "conv16", 32, 32, 16, 32, 3, 2, 1, gamma=2),
        # ResNet-18 at N = 2^15, one batched call of two uneven rounds: the
        # strided conv that opens the last stage and the classifier (with the
        # average pool folded in).
        {"name": "resnet18_batch", "kind": "batch", "params": "r18", "layers": "8x8 fc200 + 16x16x256->512 /2"},
        # ResNet-34's classifier at N = 2^16: 25088 taps in each of 1000
        # outputs (a ragged group of 1024).
        conv_round("resnet34_fc", "r34", 7, 7, 512, 1000, 7, 1, 0),
        # ResNet-34 at N = 2^16, the first conv of its last stage: the largest
        # call, 25088 outputs and 32768 key switches.
        conv_round("resnet34_conv", "r34", 14, 14, 256, 512, 3, 2, 1),
        # The transform as a call of its own: a large forward batch at the
        # largest ring, and an odd-sized inverse batch at N = 2^14.
        {"name": "ntt_forward_2e16", "kind": "ntt", "params": "r34", "count": 512, "inverse": False},
        {"name": "ntt_inverse_2e14", "kind": "ntt", "params": "conv16", "count": 37, "inverse": True},
        # Prime-power rings of Table 2: the transform at M = 3^7, and an
        # odd-sized RNS key switch at M = 5^5.
        {"name": "pp_ntt_3e7", "kind": "pp_ntt", "t": 3, "alpha": 7, "limbs": 5, "count": 4096, "inverse": False},
        {"name": "pp_keyswitch_5e5", "kind": "pp_ks", "t": 5, "alpha": 5, "limbs": 3, "count": 333, "h": 6},
        # The paper's torus scheme at its largest ring: one launch over a batch
        # of ciphertexts, as each step of its homomorphic trace does.
        {"name": "torus_keyswitch_5e5", "kind": "tq_ks", "t": 5, "alpha": 5, "D": 310, "l": 5, "count": 4096, "h": 2},
    ]


def conv_round(name, params, H, W, C_in, C_out, k, stride, pad, gamma=0):
    return {"name": name, "kind": "round", "params": params, "H": H, "W": W, "C_in": C_in, "C_out": C_out, "k": k,
            "stride": stride, "pad": pad, "gamma": gamma}


def draw(rng):
    """One more case of the same ranges (see the listed ones)."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("round", "round", "round", "rotate", "ntt", "pp_ntt", "pp_ks", "tq_ks"))
    if kind == "round":
        # convolutions of the shapes of the networks' stages, odd sizes among
        # them; outputs from a handful to half a slot-full ring
        params = rng.choice(("fc64", "conv16", "conv16", "r18", "r34"))
        most = {"fc64": 8192, "conv16": 16384, "r18": 16384, "r34": 8192}[params]
        k, stride = rng.choice(((1, 1), (3, 1), (3, 2)))
        side = log_int(1 if k == 1 else 3, 28)
        H, W = side, max(1 if k == 1 else 3, side + rng.choice((-1, 0, 0, 2)))
        pad = k // 2
        area = ((H + 2 * pad - k) // stride + 1) * ((W + 2 * pad - k) // stride + 1)
        C_out = log_int(1, max(2, min(512, most // area)))
        while C_out > 1 and C_out * area > most:
            C_out -= 1
        C_in = log_int(1, min(256, max(2, 2 * (1 << wl.PARAMS[params].log_n) // (H * W))))
        gamma = rng.choice((0, 0, 2)) if C_out * area > 1 else 0
        c = conv_round("", params, H, W, C_in, C_out, k, stride, pad, gamma)
        del c["name"]
        return c
    if kind == "rotate":
        params = rng.choice(("fc64", "conv16", "r18", "r34"))
        log_n = wl.PARAMS[params].log_n
        return {"kind": "rotate", "params": params, "count": log_int(1, 300), "d": (1 << rng.randint(1, log_n)) + 1}
    if kind == "ntt":
        params = rng.choice(("fc64", "conv16", "r18", "r34"))
        return {"kind": "ntt", "params": params, "count": log_int(1, 512), "inverse": rng.random() < 0.5}
    t, alpha = rng.choice(((3, 7), (7, 4), (5, 5)))
    if kind == "pp_ntt":
        return {"kind": "pp_ntt", "t": t, "alpha": alpha, "limbs": rng.randint(1, 5), "count": log_int(1, 4096),
                "inverse": rng.random() < 0.5}
    if kind == "pp_ks":
        return {"kind": "pp_ks", "t": t, "alpha": alpha, "limbs": rng.randint(1, 4), "count": log_int(1, 512),
                "h": 1 + t}
    t, alpha, D, l = rng.choice(TORUS)
    return {"kind": "tq_ks", "t": t, "alpha": alpha, "D": D, "l": l, "count": log_int(1, 4096), "h": 2}


# ------------------------------------------------------------------ layers --

def layer_case(case, seed):
    """The round of a `round` case: seeded weights, an input U(0, 1) (a
    post-ReLU activation) and random input and output permutations."""
    rng = np.random.default_rng((seed, 1))
    t = wl.Term(0, case["H"], case["W"], case["C_in"], case["C_out"], case["k"], case["k"], case["stride"], case["pad"])
    if case["k"] == case["H"] == case["W"] and case["k"] > 3:
        # a classifier with the global average pool folded into its kernel
        w = wl.kaiming_uniform(rng, (t.C_out, 1, 1, t.C_in), t.C_in) / (t.kh * t.kw)
        w = np.broadcast_to(w, (t.C_out, t.kh, t.kw, t.C_in)).copy()
    else:
        w = wl.kaiming_uniform(rng, (t.C_out, t.kh, t.kw, t.C_in), t.fan_in)
    x = rng.uniform(0.0, 1.0, t.H * t.W * t.C_in)
    sp = wl.random_permutation(rng, x.size)
    so = wl.random_permutation(rng, t.H_out * t.W_out * t.C_out)
    return wl.LayerCase("round", [t], [w], None, x, sp, so)


def batch_shapes():
    """The two rounds of the ResNet-18 batch: the strided conv that opens the
    last stage, and the classifier."""
    return [conv_round("", "r18", 16, 16, 256, 512, 3, 2, 1), conv_round("", "r18", 8, 8, 512, 200, 8, 1, 0)]


class _Handle:
    """A library handle, destroyed with the last reference to it (the
    references in `uses` keep what it depends on alive until then)."""

    def __init__(self, value, destroy, *uses):
        self.value = value
        weakref.finalize(self, _destroy, destroy, value, uses)


def _destroy(destroy, value, uses):
    destroy(value)


@functools.lru_cache(maxsize=1)
def _context(name):
    """One context per parameter set, as a server keeps it for every request
    (the tables and the workspace belong to it); the last one asked for stays."""
    ps = wl.PARAMS[name]
    params = _Handle(sf.sf_params_create(ps.log_n, ps.n_data, ps.data_bits, ps.n_special, ps.special_bits, ps.sigma),
                     sf.sf_params_destroy)
    return _Handle(sf.sf_ctx_create(params.value, torch.cuda.current_device()), sf.sf_ctx_destroy, params), params


def _residues(shape_head, moduli, n, seed):
    """Uniform residues [*shape_head][limb][n] on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty((*shape_head, len(moduli), n), dtype=torch.int64, device="cuda")
    for i, q in enumerate(moduli):
        out[..., i, :] = torch.randint(0, q, (*shape_head, n), generator=g, device="cuda", dtype=torch.int64)
    return out


def _prepare_round(case, seed, ctx, params, sk, ps):
    """Encrypted input, encoded weights and output buffer of one round."""
    lc = layer_case(case, seed)
    n, L = 1 << ps.log_n, ps.n_data
    layer = _Handle(sf.sf_encode_weights(ctx.value, lc.terms, lc.weights[0], None, ps.delta, ps.delta ** 2),
                    sf.sf_layer_destroy, ctx)
    info = sf.sf_layer_get_info(ctx.value, layer.value)
    k_in = info["k_in"]
    msg = sf.sf_encode_input(lc.x[lc.sigma_prev.astype(np.int64)], ps.delta)
    d_in = torch.empty((k_in, 2, L, n), dtype=torch.int64, device="cuda")
    sf.sf_encrypt(ctx.value, sk.value, msg, seed * 7 + 1, d_in, k_in)
    d_pow = None
    if case["gamma"] == 2:
        d_pow = torch.empty_like(d_in)
        sf.sf_encrypt(ctx.value, sk.value, sf.sf_client_power(params.value, msg, k_in, 3), seed * 7 + 2, d_pow, k_in)
    sf.sf_sync(ctx.value)
    return {"layer": layer, "k_in": k_in, "d_in": d_in, "d_pow": d_pow, "sp": lc.sigma_prev, "so": lc.sigma_out,
            "groups": info["n_groups"], "d_out": torch.empty((info["n_groups"], 2, L, n), dtype=torch.int64, device="cuda")}


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind in ("round", "batch", "rotate", "ntt"):
        ps = wl.PARAMS[case["params"]]
        ctx, params = _context(case["params"])
        st["ctx"] = ctx
        n, L = 1 << ps.log_n, ps.n_data
        q = sf.sf_params_get_info(params.value)["moduli"][:L]
        if kind == "ntt":
            st["in"] = _residues((case["count"],), q, n, seed)
            st["out"] = torch.empty_like(st["in"])
            return st
        sk = _Handle(sf.sf_keygen(ctx.value, seed * 7 + 3), sf.sf_secret_key_destroy, ctx)
        d = [case["d"]] if kind == "rotate" else None
        st["rk"] = _Handle(sf.sf_gen_rotation_keys(ctx.value, sk.value, d, seed * 7 + 4), sf.sf_rotkeys_destroy, ctx)
        if kind == "rotate":
            # ciphertexts are uniform residues to anyone without the key
            st["in"] = _residues((case["count"], 2), q, n, seed)
            st["out"] = torch.empty_like(st["in"])
            return st
        shapes = batch_shapes() if kind == "batch" else [case]
        st["rounds"] = [_prepare_round(c, seed * 16 + i, ctx, params, sk, ps) for i, c in enumerate(shapes)]
        return st
    t, alpha, count = case["t"], case["alpha"], case["count"]
    dev = torch.cuda.current_device()
    if kind in ("pp_ntt", "pp_ks"):
        ring = _Handle(sf.sf_pp_ring_create(t, alpha, case["limbs"], 50, dev), sf.sf_pp_ring_destroy)
        info = sf.sf_pp_ring_info(ring.value, case["limbs"])
        st["ring"] = ring
        if kind == "pp_ntt":
            st["in"] = _residues((count,), info["moduli"], info["M"], seed)
            st["out"] = torch.empty_like(st["in"])
            return st
        N, Lp = info["N"], case["limbs"]
        rng = np.random.default_rng((seed, 2))
        s = torch.as_tensor(rng.integers(-1, 2, N)).cuda()
        e = torch.as_tensor(rng.integers(-3, 4, (Lp, N))).cuda()
        st["ka"] = _residues((Lp,), info["moduli"], N, seed + 1)
        st["kb"] = torch.empty_like(st["ka"])
        sf.sf_pp_ksk(ring.value, s, case["h"], st["ka"], e, st["kb"])
        st["in"] = _residues((count, 2), info["moduli"], N, seed)
        st["out"] = torch.empty_like(st["in"])
        torch.cuda.synchronize()
        return st
    ring = _Handle(sf.sf_tq_ring_create(t, alpha, case["D"], case["l"], dev), sf.sf_tq_ring_destroy)
    info = sf.sf_tq_ring_info(ring.value)
    N, l = info["N"], case["l"]
    rng = np.random.default_rng((seed, 3))
    s = torch.as_tensor(rng.integers(-1, 2, N)).cuda()
    e = torch.as_tensor(rng.integers(-(1 << 17), (1 << 17) + 1, (l, N))).cuda()
    g = torch.Generator(device="cuda").manual_seed(seed)
    ka = torch.randint(0, 1 << 53, (l, N), generator=g, device="cuda", dtype=torch.int64)
    kb = torch.empty_like(ka)
    sf.sf_tq_ksk(ring.value, s, case["h"], ka, e, kb)
    st["key"] = torch.empty(info["key_words"], dtype=torch.int64, device="cuda")
    sf.sf_tq_key_prepare(ring.value, ka, kb, st["key"])
    st["ring"] = ring
    st["in"] = torch.randint(0, 1 << 53, (count, 2, N), generator=g, device="cuda", dtype=torch.int64)
    st["out"] = torch.empty_like(st["in"])
    torch.cuda.synchronize()
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "round":
        r = st["rounds"][0]
        if c["gamma"] == 2:
            sf.sf_eval_linear_layer_gamma(st["ctx"].value, r["layer"].value, st["rk"].value, 2, r["d_in"], r["d_pow"],
                                          r["k_in"], r["sp"], r["so"], r["d_out"], r["groups"])
        else:
            sf.sf_eval_linear_layer(st["ctx"].value, r["layer"].value, st["rk"].value, r["d_in"], r["k_in"], r["sp"],
                                    r["so"], r["d_out"], r["groups"])
        return r["d_out"]
    if kind == "batch":
        rs = st["rounds"]
        sf.sf_eval_layers(st["ctx"].value, [r["layer"].value for r in rs], [st["rk"].value] * len(rs),
                          [r["d_in"] for r in rs], [r["k_in"] for r in rs], [r["sp"] for r in rs],
                          [r["so"] for r in rs], [r["d_out"] for r in rs], [r["groups"] for r in rs])
        return [r["d_out"] for r in rs]
    if kind == "rotate":
        sf.sf_rotate(st["ctx"].value, st["rk"].value, c["d"], st["in"], st["out"], c["count"])
    elif kind == "ntt":
        sf.sf_ntt_batch(st["ctx"].value, st["in"], st["out"], c["count"], c["inverse"])
    elif kind == "pp_ntt":
        sf.sf_pp_ntt(st["ring"].value, st["in"], st["out"], c["count"], c["inverse"])
    elif kind == "pp_ks":
        sf.sf_pp_keyswitch(st["ring"].value, st["in"], st["out"], c["count"], c["h"], st["ka"], st["kb"])
    else:
        sf.sf_tq_keyswitch(st["ring"].value, st["in"], st["out"], c["count"], c["h"], st["key"])
    return st["out"]


# -------------------------------------------------------------------- work --
# "flops" counts modular multiplications, two operations (multiply, add) each;
# "bytes" the call's inputs (keys among them) and outputs once each.

def _ks_products(ps):
    """Modular multiplications of one hybrid key switch: limb transforms, key
    products and base conversions."""
    n, L, K = 1 << ps.log_n, ps.n_data, ps.n_special
    dnum, nm = -(-L // K), L + K
    transforms = L + (dnum * nm - L) + 2 * K + 2 * L
    return transforms * (n // 2) * ps.log_n + 2 * dnum * nm * n + 2 * L * K * n


def _key_bytes(ps):
    L, K = ps.n_data, ps.n_special
    return (-(-L // K)) * 2 * (L + K) * 8 << ps.log_n


def _round_work(c):
    ps = wl.PARAMS[c["params"]]
    n, L = 1 << ps.log_n, ps.n_data
    Ho, Wo = (c["H"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1, (c["W"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1
    e_in, e_out = c["H"] * c["W"] * c["C_in"], Ho * Wo * c["C_out"]
    k_in = -(-e_in // n)
    ks = max(1, e_out - (e_out // 2 if c["gamma"] == 2 else 0))
    groups = -(-e_out // (n // 2))
    parts = k_in * (2 if c["gamma"] == 2 else 1)
    leaf = parts * L * ((n // 2) * ps.log_n + 2 * n)
    ct = 2 * L * n * 8
    keys = ps.log_n * _key_bytes(ps)
    return {"bytes": parts * ct + groups * ct + keys + 8 * c["C_out"] * c["k"] ** 2 * c["C_in"],
            "flops": 2 * (e_out * leaf + ks * _ks_products(ps))}


def work(case):
    kind = case["kind"]
    if kind == "round":
        return _round_work(case)
    if kind == "batch":
        ws = [_round_work(c) for c in batch_shapes()]
        keys = wl.PARAMS["r18"].log_n * _key_bytes(wl.PARAMS["r18"])
        return {"bytes": sum(w["bytes"] for w in ws) - keys, "flops": sum(w["flops"] for w in ws)}
    if kind in ("rotate", "ntt"):
        ps = wl.PARAMS[case["params"]]
        n, L = 1 << ps.log_n, ps.n_data
        if kind == "ntt":
            return {"bytes": 2 * case["count"] * L * n * 8, "flops": 2 * case["count"] * L * (n // 2) * ps.log_n}
        return {"bytes": 2 * case["count"] * 2 * L * n * 8 + _key_bytes(ps), "flops": 2 * case["count"] * _ks_products(ps)}
    t, alpha, count = case["t"], case["alpha"], case["count"]
    M = t ** alpha
    N = M - M // t
    transform = alpha * (M // t) * ((t - 1) + max(2, (t - 1) ** 2 // 2))
    if kind == "pp_ntt":
        polys = count * case["limbs"]
        return {"bytes": 2 * polys * M * 8, "flops": 2 * polys * transform}
    if kind == "pp_ks":
        L = case["limbs"]
        return {"bytes": (2 * count * 2 * L + 2 * L * L) * N * 8, "flops": 2 * count * ((L * L + 2 * L) * transform + 2 * L * L * M)}
    l = case["l"]
    return {"bytes": 2 * count * 2 * N * 8 + 8 * l * M * 8, "flops": 2 * count * (2 * (l + 2) * transform + 4 * l * M)}


def exact(case, seed):
    """Outputs are whole numbers, compared bit for bit; none is a rounded value."""
    return None
