"""The backward's dW + dH launch at the shapes where its tiling can go wrong,
every gradient entry against the fp64 oracle (max-norm bound of helpers.py:
bf16 rounding of dL/dz and, for fp32 storage, tf32 products, 2^-10 relative
each, stay far below it)."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2608_09703_gb300 import binding as B
from paper_2608_09703_gb300 import synth

from helpers import check_forward, check_grads, run_gpu

pytestmark = pytest.mark.gpu


def grads_match_oracle(wl, seed, vocab_group=0):
    H, W, y = synth.make_inputs(wl, seed=seed)
    y[0] = -1
    op, status = run_gpu(wl, H, W, y, grad_scale=1.3, vocab_group=vocab_group)
    assert status == 0, B.mls_strerror(status)
    Ho, Wo = synth.as_oracle_arrays(H), synth.as_oracle_arrays(W)
    yo = y.cpu().numpy().astype(np.int32)
    kw = dict(teacher=wl.teacher_index, tau=wl.tau, alpha=wl.alpha, w=wl.weights)
    check_forward(op, oracle.forward(Ho, Wo, yo, **kw))
    dH, dW = oracle.backward(Ho, Wo, yo, grad_scale=1.3, **kw)
    check_grads(op, dH=dH, dW=dW)
    return op


@pytest.mark.parametrize("T,d,V,vocab_group", [
    (300, (36, 100), 1003, 0),       # widths, tokens and vocabulary that end inside a 32-wide block
    (257, (256, 516), 700, 256),     # three vocabulary groups, dH accumulated
    (40, (512, 1024), 17000, 0),     # dH over more than 512 k-blocks of 32, 7 units each
])
def test_fp32_reads_g_h_w_in_place(T, d, V, vocab_group):
    """fp32 storage: both products read G, H and W transposed or not where they
    lie (no K-major copies), in one launch."""
    wl = synth.Workload("fp32", T=T, d=d, V=V, dtype="fp32", tau=0.8, alpha=0.4, w_sigma=0.05)
    grads_match_oracle(wl, seed=21, vocab_group=vocab_group)


@pytest.mark.parametrize("dtype,T,d,V,vocab_group", [
    ("bf16", 70, (64, 136), 20000, 0),      # dH: 2 tiles over 313 k-blocks
    ("bf16", 70, (64, 136), 20011, 9984),   # three groups: the copies added to dH
    ("fp32", 33, (36, 100), 9001, 0),
    ("bf16", 9001, (64, 136), 300, 0),      # dW: 4 tiles over 141 k-blocks of tokens
    ("fp32", 5000, (36, 100), 257, 0),
])
def test_split_reduction(dtype, T, d, V, vocab_group):
    """A few long reductions, cut into several units each: the last split
    shorter than the others, and the copies summed into the output."""
    wl = synth.Workload("split", T=T, d=d, V=V, dtype=dtype, tau=0.8, alpha=0.4, w_sigma=0.05)
    B.mls_profile_enable(True)
    try:
        grads_match_oracle(wl, seed=22, vocab_group=vocab_group)
        assert "split_sum" in B.mls_profile_read()
    finally:
        B.mls_profile_enable(False)
