"""dH in wide units: a vocabulary group that writes dH over at least 512 k-blocks
of the vocabulary, with an even number of column tiles in every sub-model, runs
pairs of column tiles that share each A tile of G.  Shorter or fewer reductions
are split instead, so these shapes have enough token tiles to stay whole: widths
of 2 and 4 column tiles (the last ragged) over 11 or 13 token tiles (the last
ragged), with a second group that runs plain and accumulates into dH, in both
storage types.  Every entry of every gradient against fp64 torch on the device
(the oracle needs minutes here)."""
import pytest
import torch

from paper_2608_09703_gb300 import binding as B
from paper_2608_09703_gb300 import synth

from helpers import launch_plan, run_gpu

D = (264, 776)
# dtype, T, V, vocab_group, units of the groups
CASES = [("bf16", 2700, 33000, 0, [1]),
         ("bf16", 2700, 66000, 33024, [1, 0]),
         ("fp32", 3100, 16800, 0, [1]),
         ("fp32", 3100, 34000, 17152, [1, 0])]


def workload(dtype, T, V):
    return synth.Workload("wide", T=T, d=D, V=V, dtype=dtype, tau=1.3, alpha=0.5, w_sigma=0.05)


@pytest.mark.parametrize("dtype,T,V,vocab_group,wide", CASES)
def test_plan(dtype, T, V, vocab_group, wide):
    plan = launch_plan(workload(dtype, T, V), vocab_group)
    assert plan["wide"] == wide and plan["ksplit"] == [1] * len(wide)


def exact_grads(H, W, y, tau, alpha, scale):
    """Gradients of scale * loss (teacher: the last sub-model, weights 1) in fp64."""
    T, n = H[0].shape[0], int((y >= 0).sum())
    Hd, Wd = [h.double() for h in H], [w.double() for w in W]
    dH, dW = [torch.zeros_like(h) for h in Hd], [torch.zeros_like(w) for w in Wd]
    for a in range(0, T, 512):
        rows = slice(a, min(a + 512, T))
        ok = y[rows] >= 0
        idx = y[rows].clamp(min=0).long()[:, None]
        q = torch.softmax(Hd[-1][rows] @ Wd[-1].T / tau, -1)
        for m in range(len(H)):
            z = Hd[m][rows] @ Wd[m].T
            G = torch.softmax(z, -1)
            G.scatter_add_(-1, idx, torch.full_like(idx, -1, dtype=torch.float64))
            if m + 1 < len(H):
                G.mul_(1 - alpha).add_(torch.softmax(z / tau, -1) - q, alpha=alpha / tau)
            G *= torch.where(ok, scale / n, 0.0)[:, None]
            dH[m][rows] = G @ Wd[m]
            dW[m] += G.T @ Hd[m][rows]
    return dH, dW


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,T,V,vocab_group,wide", CASES)
def test_gradients(dtype, T, V, vocab_group, wide):
    wl = workload(dtype, T, V)
    plan = launch_plan(wl, vocab_group)
    assert plan["wide"] == wide, plan
    H, W, y = synth.make_inputs(wl, seed=13, device="cuda")
    y[[0, 300, T - 1]] = -1
    B.mls_profile_enable(True)
    try:
        op, status = run_gpu(wl, H, W, y, grad_scale=1.7, vocab_group=vocab_group)
        assert "split_sum" not in B.mls_profile_read()
    finally:
        B.mls_profile_enable(False)
    assert status == 0, B.mls_strerror(status)
    dH, dW = exact_grads(H, W, y, wl.tau, wl.alpha, 1.7)
    for name, got, want in (("dH", op.dH, dH), ("dW", op.dW, dW)):
        for m in range(len(D)):
            # per row of dH and per tensor of dW, 2-norms: dL/dz is rounded to bf16, or the
            # products' operands to tf32, at most 2^-9 relative each; 2^-7 leaves room for
            # the logits' own rounding and for rows whose terms cancel in part
            err, size = (got[m] - want[m]), want[m]
            if name == "dH":
                assert torch.equal(err[y < 0], torch.zeros_like(err[y < 0]))
                rel = err[y >= 0].norm(dim=-1) / size[y >= 0].norm(dim=-1)
            else:
                rel = err.norm() / size.norm()
            assert rel.max() < 2.0 ** -7, f"{name}[{m}] {rel.max().item()}"
