"""sf_linear_outputs holds its leaves once: the context's workspace grows by the
leaves, the leaf launches' scratch and small change, not by a second copy."""
import numpy as np
import pytest
import torch

import paper_2509_01253_gb300 as sf
from paper_2509_01253_gb300 import workloads as wl
from _gpu import Session, dev_zeros, from_dev, gpu_layer, stream_input

pytestmark = pytest.mark.gpu


def test_outputs_hold_their_leaves_once():
    case = wl.fc_case(81, 300, 1200)
    s = Session(14, 3, 50, 1, sk_seed=82, rot=False)
    try:
        lay = gpu_layer(s, case, 2.0 ** 20, 2.0 ** 40)
        d_in = s.encrypt(sf.sf_encode_input(stream_input(case), 2.0 ** 20), 83, 1)
        few, out = dev_zeros(2, 2, s.L, s.n), dev_zeros(1200, 2, s.L, s.n)
        sf.sf_linear_outputs(s.ctx, lay, d_in, 1, case.sigma_prev, np.array([0, 1199]), few)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        sf.sf_linear_outputs(s.ctx, lay, d_in, 1, case.sigma_prev, np.arange(1200), out)
        torch.cuda.synchronize()
        used = free - torch.cuda.mem_get_info()[0]
        leaves = 1200 * 2 * s.L * s.n * 8
        # column-pass scratch and tap buckets of a leaf launch: at most 256 MiB each
        # (300 taps of 16 bytes a slot); the pool grows by an eighth more
        assert used <= (leaves + (256 << 20) + 1200 * 300 * 16 + (16 << 20)) * 9 / 8
        assert (from_dev(out)[[0, 1199]] == from_dev(few)).all()
        sf.sf_layer_destroy(lay)
    finally:
        s.close()
