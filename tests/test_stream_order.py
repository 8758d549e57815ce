"""The kernels of a call are chained with programmatic dependent launches, each
allowed to start before its predecessor has finished.  Their order has to hold
between back-to-back calls that share buffers and workspace, against other work
on the stream, and in a captured graph."""
import pytest
import torch

from paper_2608_09703_gb300 import binding as B
from paper_2608_09703_gb300 import synth

pytestmark = pytest.mark.gpu


def _op(T, d, V, vocab_group, seed):
    wl = synth.Workload("order", T=T, d=d, V=V, tau=0.9, alpha=0.4, w_sigma=0.05)
    H, W, y = synth.make_inputs(wl, seed=seed, device="cuda")
    return B.HeadLoss(d, T, V, tau=0.9, alpha=0.4, vocab_group=vocab_group), H, W, y


def _outputs(op):
    return [t.clone() for t in (op.loss, op.tok_loss, op.stats, *op.dH, *op.dW)]


# several groups (dH accumulated), split reductions, a plain small step
@pytest.mark.parametrize("T,d,V,vocab_group", [(300, (64, 136), 3000, 768), (70, (64, 136), 20000, 0),
                                               (513, (64, 136), 1000, 0)])
def test_back_to_back_calls_and_graph(T, d, V, vocab_group):
    op, H, W, y = _op(T, d, V, vocab_group, 3)
    _, H2, W2, y2 = _op(T, d, V, vocab_group, 4)
    want = []
    for h, w, t in ((H, W, y), (H2, W2, y2)):
        op.forward(h, w, t)
        op.backward(h, w, t)
        torch.cuda.synchronize()
        want.append(_outputs(op))
    # inputs that change on the stream right before each call, no host synchronisation
    Hc, Wc, yc = [h.clone() for h in H], [w.clone() for w in W], y.clone()
    got = []
    for i in range(20):
        h, w, t = ((H, W, y), (H2, W2, y2))[i % 2]
        for a, b in zip(Hc + Wc + [yc], list(h) + list(w) + [t]):
            a.copy_(b)
        op.forward(Hc, Wc, yc)
        op.backward(Hc, Wc, yc)
        got.append(_outputs(op))
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(g, want[i % 2])), f"call {i}"
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            op.forward(Hc, Wc, yc)
            op.backward(Hc, Wc, yc)
    for i in (0, 1, 0):
        h, w, t = ((H, W, y), (H2, W2, y2))[i]
        for a, b in zip(Hc + Wc + [yc], list(h) + list(w) + [t]):
            a.copy_(b)
        for out in op.dH + op.dW + [op.loss, op.tok_loss]:
            out.fill_(7.0)
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(_outputs(op), want[i]))
    assert B.mls_get_status() == 0


@pytest.mark.parametrize("b,greedy", [(3, False), (60, False), (3, True)])
def test_spec_and_pairwise_back_to_back(b, greedy):
    wl = synth.SpecWorkload("order", B=b, gamma=4, V=9000, d_draft=64, d_verify=136)
    sets = []
    for seed in (1, 2):
        Hd, Wd, Hv, Wv = synth.make_spec_inputs(wl, seed, device="cuda")
        draft = (Hd.float() @ Wd.float().T).argmax(-1).to(torch.int32).view(b, 4)
        sets.append((Hd, Wd, Hv, Wv, draft, synth.make_uniforms(b, 4, seed, device="cuda")))
    op = B.SpecVerify(b, 4, wl.V, 64, 136, greedy=greedy)
    pair = B.HeadLoss((64, 136), b * 4, wl.V)
    want = []
    for x in sets:
        n = [t.clone() for t in op(*x)]
        H = [x[0], torch.cat([x[0], x[0], x[0][:, :8]], 1)]
        want.append(n + [t.clone() for t in pair.pairwise(H, [x[1], x[3]])])
        torch.cuda.synchronize()
    got = []
    for i in range(20):
        x = sets[i % 2]
        H = [x[0], torch.cat([x[0], x[0], x[0][:, :8]], 1)]
        got.append([t.clone() for t in op(*x)] + [t.clone() for t in pair.pairwise(H, [x[1], x[3]])])
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert all(torch.equal(a, c) for a, c in zip(g, want[i % 2])), f"call {i}"
