"""Token tiles and vocabularies for which a head or evaluation launch leaves some
vocabulary tiles to extra pairs (76 resident pairs: 6 token tiles x 12 splits and
12 x 6 leave four pairs' SMs free), against the oracle.  The plan of every shape
is asserted: each runs as well, unnoticed, without extra pairs."""
import pytest
import torch

from paper_2608_09703_gb300 import binding as B
from paper_2608_09703_gb300 import synth

from helpers import exact_logits, launch_plan
from test_backward_gemm import grads_match_oracle

# dtype, T, d, V, vocab_group, extra pairs per token tile in the forward and in each backward group
STEPS = [("bf16", 1531, (64, 136), 32003, 0, 2, [2]),          # 126 tiles: runs of 3, the last one ragged
         ("bf16", 1290, (72, 64, 80), 38269, 19200, 2, [3, 3]),  # two groups of 75 tiles, runs of 1
         ("fp32", 1300, (36, 68), 22173, 0, 1, [1])]           # 87 tiles: a run of 3, the last one ragged
# dtype, d, T, V, extra pairs per token tile
EVALS = [("bf16", (64, 136), 2999, 20011, 1),
         ("bf16", (72, 64, 80), 1290, 25523, 2), ("fp32", (36, 68, 72), 1290, 25523, 2),
         ("bf16", (64, 72, 80, 88), 1290, 12723, 2)]           # 100 tiles of 128 columns


def step_workload(dtype, T, d, V):
    return synth.Workload("extra", T=T, d=d, V=V, dtype=dtype, tau=0.8, alpha=0.4, w_sigma=0.05,
                          teacher=0)


def eval_workload(dtype, d, T, V):
    return synth.Workload("extra", T=T, d=d, V=V, dtype=dtype, w_sigma=0.05)


def test_plans():
    for dtype, T, d, V, vocab_group, fwd, bwd in STEPS:
        plan = launch_plan(step_workload(dtype, T, d, V), vocab_group)
        assert plan["fwd_extra"] == fwd and plan["bwd_extra"] == bwd, (dtype, T, V, plan)
    for dtype, d, T, V, extra in EVALS:
        plan = launch_plan(eval_workload(dtype, d, T, V))
        assert plan["eval_extra"] == extra, (dtype, d, V, plan)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,T,d,V,vocab_group,fwd,bwd", STEPS)
def test_step(dtype, T, d, V, vocab_group, fwd, bwd):
    wl = step_workload(dtype, T, d, V)
    plan = launch_plan(wl, vocab_group)
    assert plan["fwd_extra"] == fwd and plan["bwd_extra"] == bwd, plan
    grads_match_oracle(wl, seed=24, vocab_group=vocab_group)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d,T,V,extra", EVALS)
def test_pairwise(dtype, d, T, V, extra):
    wl = eval_workload(dtype, d, T, V)
    assert launch_plan(wl)["eval_extra"] == extra
    H, W, y = synth.make_inputs(wl, seed=25)
    y[[3, T - 1]] = -1
    op = B.HeadLoss(d, T, V, dtype=H[0].dtype)
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
