"""The key-switch workspace of a round: (dnum + 2)(L + K) + L limbs per merge of a
launch batch, from the growth of the context's pool with the batch."""
import pytest
import torch

import paper_2509_01253_gb300 as sf
from paper_2509_01253_gb300 import workloads as wl
from _gpu import Session, dev_zeros, from_dev, gpu_layer, stream_input

pytestmark = pytest.mark.gpu


def test_workspace_per_merge():
    log_n, L, K, merges = 12, 6, 1, 256   # 512 outputs: 256 merges in the widest level
    case = wl.fc_case(31, 64, 2 * merges)
    used, outs = [], []
    for batch in (1, merges):
        s = Session(log_n, L, 50, K, sk_seed=32, rk_seed=33)
        try:
            sf.sf_ctx_set_option(s.ctx, "ks_batch", batch)
            sf.sf_ctx_set_option(s.ctx, "use_graph", 0)
            lay = gpu_layer(s, case, 2.0 ** 20, 2.0 ** 40)
            d_in = s.encrypt(sf.sf_encode_input(stream_input(case), 2.0 ** 20), 34, 1)
            out = dev_zeros(1, 2, L, s.n)
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            sf.sf_eval_linear_layer(s.ctx, lay, s.rk, d_in, 1, case.sigma_prev, case.sigma_out, out, 1)
            sf.sf_sync(s.ctx)
            used.append(free - torch.cuda.mem_get_info()[0])
            outs.append(from_dev(out))
            sf.sf_layer_destroy(lay)
        finally:
            s.close()
    assert (outs[0] == outs[1]).all()
    dnum = -(-L // K)
    limbs = (dnum + 2) * (L + K) + L
    # the pool grows by an eighth more than asked; allocations come in 2 MiB pages
    assert used[1] - used[0] <= (merges - 1) * limbs * s.n * 8 * 9 / 8 + (8 << 20)
