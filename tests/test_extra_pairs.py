"""Token tiles and vocabularies for which a head or evaluation launch leaves some
vocabulary tiles to extra pairs (76 resident pairs: 6 token tiles x 12 splits and
12 x 6 leave four pairs' SMs free), against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2608_09703_gb300 import binding as B
from paper_2608_09703_gb300 import synth

from helpers import exact_logits
from test_backward_gemm import grads_match_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,T,d,V,vocab_group", [
    ("bf16", 1531, (64, 136), 32003, 0),       # 126 tiles: runs of 3, the last one ragged
    ("bf16", 1290, (72, 64, 80), 32003, 16128),  # the same in two groups of 63 tiles
    ("fp32", 1300, (36, 68), 20011, 0),
])
def test_step(dtype, T, d, V, vocab_group):
    wl = synth.Workload("extra", T=T, d=d, V=V, dtype=dtype, tau=0.8, alpha=0.4, w_sigma=0.05,
                        teacher=0)
    grads_match_oracle(wl, seed=24, vocab_group=vocab_group)


@pytest.mark.parametrize("d,T,V", [((64, 136), 2999, 20011), ((72, 64, 80), 1290, 32003),
                                   ((64, 72, 80, 88), 1290, 16003)])
def test_pairwise(d, T, V):
    wl = synth.Workload("extra", T=T, d=d, V=V, w_sigma=0.05)
    H, W, y = synth.make_inputs(wl, seed=25)
    y[[3, T - 1]] = -1
    op = B.HeadLoss(d, T, V)
    kl, am, stats = op.pairwise([h.cuda() for h in H], [w.cuda() for w in W], y.cuda())
    torch.cuda.synchronize()
    assert B.mls_get_status() == 0
    z = exact_logits(H, W)
    for i in range(len(d)):
        for j in range(len(d)):
            pi, pj = torch.log_softmax(z[i], -1), torch.log_softmax(z[j], -1)
            want = (pi.exp() * (pi - pj)).sum(-1)
            # fp32 sums over V terms in tiles, KL of order 0.1: 1e-3 of max(1, KL) as in helpers.py
            assert (kl[i, j].cpu().double() - want).abs().max() < 1e-3
            ok = y >= 0
            assert abs(stats[0, i, j].item() - want[ok].mean().item()) < 1e-3
