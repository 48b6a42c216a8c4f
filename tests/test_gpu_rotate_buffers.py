"""Rotations whose output shares words with their input: in place, and shifted
by one ciphertext either way, in one launch batch and in several, by both entry
points, equal word for word to the same rotation between separate buffers
(which other tests compare with the oracle)."""
import pytest
import torch

import paper_2509_01253_gb300 as sf
from _gpu import Session, dev_zeros, from_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rotate", [sf.sf_rotate, sf.sf_rotate_noalloc])
@pytest.mark.parametrize("log_n,L,K,count,ks_batch", [(10, 3, 1, 1, 512), (12, 4, 2, 5, 512), (12, 4, 2, 5, 2), (14, 3, 1, 7, 512)])
def test_rotation_onto_its_input(rotate, log_n, L, K, count, ks_batch):
    n = 1 << log_n
    s = Session(log_n, L, 50, K, sk_seed=91, rk_seed=92, rot_d=[5])
    try:
        sf.sf_ctx_set_option(s.ctx, "ks_batch", ks_batch)
        x = s.encrypt([k % 1000 for k in range(count * n)], 93, count)
        want = dev_zeros(count, 2, L, n)
        sf.sf_rotate(s.ctx, s.rk, 5, x, want, count)
        for shift in (0, 1, -1):   # output `shift` ciphertexts after the input
            buf = dev_zeros(count + 2, 2, L, n)
            buf[1:count + 1] = x
            rotate(s.ctx, s.rk, 5, buf[1:], buf[1 + shift:], count)
            sf.sf_sync(s.ctx)
            assert (from_dev(buf[1 + shift:count + 1 + shift]) == from_dev(want)).all(), shift
    finally:
        s.close()


@pytest.mark.parametrize("rotate", [sf.sf_rotate, sf.sf_rotate_noalloc])
@pytest.mark.parametrize("count", [1, 3])
def test_captured_in_place(rotate, count):
    """The copy and the key switch in a caller's graph, replayed on new contents."""
    s = Session(11, 3, 50, 1, sk_seed=94, rk_seed=95, rot_d=[9])
    try:
        xs = [s.encrypt([k % m for k in range(count * s.n)], m, count) for m in (101, 102)]
        want = [dev_zeros(count, 2, 3, s.n) for _ in xs]
        for x, w in zip(xs, want):
            sf.sf_rotate(s.ctx, s.rk, 9, x, w, count)
        buf = xs[0].clone()
        rotate(s.ctx, s.rk, 9, buf, buf, count)   # the workspace grows outside the capture
        torch.cuda.synchronize()
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            rotate(s.ctx, s.rk, 9, buf, buf, count, stream.cuda_stream)
        for x, w in zip(xs, want):
            buf.copy_(x)
            graph.replay()
            torch.cuda.synchronize()
            assert (from_dev(buf) == from_dev(w)).all()
        sf.sf_sync(s.ctx)
    finally:
        s.close()
