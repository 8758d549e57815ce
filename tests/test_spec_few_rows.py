"""The verify step's logits for few rows (at most 128 verify positions): the row
counts at the edges of that kernel's range and just past it, a vocabulary that
ends inside a tile, and more tiles than SMs, against the oracle as in
test_spec.py."""
import pytest
import torch

from paper_2608_09703_gb300 import binding as B
from paper_2608_09703_gb300 import synth

from test_spec import check, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("greedy", [False, True])
@pytest.mark.parametrize("b,gamma,V", [(1, 1, 77), (1, 6, 1003), (2, 15, 700), (3, 10, 513),
                                       (16, 7, 1000), (43, 2, 1000)])
def test_row_counts(b, gamma, V, greedy, dtype):
    """2, 7, 32, 33, 128 and 129 verify rows (the last takes the pair GEMM)."""
    wl = synth.SpecWorkload("rows", B=b, gamma=gamma, V=V, d_draft=72, d_verify=136, dtype=dtype)
    check(wl, *inputs(wl, 31 + b), greedy=greedy, min_checked=0.5)


def test_more_tiles_than_sms_and_wide_draft():
    """469 tiles per head over 152 CTAs, and a draft wider than its verifier,
    whose tiles then go first; every row's statistics against torch."""
    for dd, dv in ((64, 136), (264, 72)):
        V, b, gamma = 60000, 3, 4
        g = torch.Generator().manual_seed(dd)
        r = lambda *s: torch.randn(*s, generator=g).to(torch.bfloat16).cuda()
        Hd, Wd, Hv, Wv = r(b * gamma, dd), r(V, dd) * 0.1, r(b * (gamma + 1), dv), r(V, dv) * 0.1
        draft = torch.randint(0, V, (b, gamma), generator=g, dtype=torch.int32).cuda()
        u = torch.rand(b, gamma + 1, 2, generator=g).cuda()
        op = B.SpecVerify(b, gamma, V, dd, dv)
        op(Hd, Wd, Hv, Wv, draft, u)
        torch.cuda.synchronize()
        assert B.mls_get_status() == 0
        tiles, ldz = -(-V // 128), -(-V // 4) * 4
        ws, off = op.ws, 0

        def take(shape):  # the workspace's layout: e_t and statistics of both sub-models
            nonlocal off
            n = 4 * shape[0] * shape[1]
            t = ws[off:off + n].view(torch.float32).view(shape)
            off += -(-n // 256) * 256
            return t
        Pv, Pd = b * (gamma + 1), b * gamma
        e = take((Pv, ldz)), take((Pd, ldz))
        st = take((Pv, 2 * tiles)), take((Pd, 2 * tiles))
        for H, W, ee, ss in ((Hv, Wv, e[0], st[0]), (Hd, Wd, e[1], st[1])):
            z = torch.full((H.shape[0], tiles * 128), float("-inf"), device="cuda", dtype=torch.float64)
            z[:, :V] = H.double() @ W.double().T
            z = z.view(H.shape[0], tiles, 128)
            m = z.amax(-1)
            want = ((z - m[..., None]) / 0.4).exp()
            # logits: fp32 sums of at most 264 exact products, |z| <= 20: 1e-5 absolute,
            # so e is right to 5e-5 relative
            assert (ss[:, 0::2].double() - m).abs().max() < 1e-4
            assert ((ss[:, 1::2].double() / want.sum(-1)) - 1).abs().max() < 1e-4
            assert (ee[:, :V].double() - want.view(H.shape[0], -1)[:, :V]).abs().max() < 1e-4


@pytest.mark.parametrize("b,V,z_std,temperature,top_p", [
    (2, 60000, 2.5, 0.9, 0.95),    # thousands of tokens in the boundary's octave: listed
    (2, 60000, 0.5, 1.0, 0.9),     # over 4096 of them: bisected first
    (2, 3000, 2.5, 0.05, 0.5),     # one token above 2^-8 settles it
    (2, 3000, 0.0, 1.0, 0.9),      # every token tied at the maximum
    (60, 9000, 2.5, 0.9, 0.99),    # 8 and 16 warps per row instead of 32
    (200, 9000, 2.5, 0.9, 0.99),
])
def test_nucleus_boundary(b, V, z_std, temperature, top_p):
    """Each row's nucleus state against fp64 sums of the stored probabilities e:
    the mass above the boundary b stays below top_p of the total, the mass from
    b on reaches it (to 1e-5, fp32 sums of at most 60000 terms in trees), and
    the ties are counted exactly."""
    gamma, dd, dv = 1, 64, 128
    wl = synth.SpecWorkload("n", B=b, gamma=gamma, V=V, d_draft=dd, d_verify=dv, z_std=z_std)
    Hd, Wd, Hv, Wv = (t.cuda() for t in synth.make_spec_inputs(wl, 5))
    op = B.SpecVerify(b, gamma, V, dd, dv, temperature=temperature, top_p=top_p)
    draft = torch.zeros(b, gamma, dtype=torch.int32, device="cuda")
    op(Hd, Wd, Hv, Wv, draft, synth.make_uniforms(b, gamma, 5).cuda())
    torch.cuda.synchronize()
    assert B.mls_get_status() == 0
    Pv, Pd = b * (gamma + 1), b * gamma
    sh = 7 if Pv <= 128 else 8
    tiles, ldz = -(-V // (1 << sh)), -(-V // 4) * 4
    off, parts = 0, []
    for rows, cols in ((Pv, ldz), (Pd, ldz), (Pv, 2 * tiles), (Pd, 2 * tiles), (Pv, tiles),
                       (Pd, tiles), (Pv, 8), (Pd, 8)):
        n = 4 * rows * cols
        parts.append(op.ws[off:off + n].view(torch.float32).view(rows, cols))
        off += -(-n // 256) * 256
    ev, ed, _, _, fv, fd, sv, sd = parts
    for e, f, st in ((ev, fv, sv), (ed, fd, sd)):
        e = e[:, :V] * f[:, torch.arange(V, device="cuda") >> sh]  # fp32, as the kernel forms it
        bound, kept = st[:, 1], st[:, 2].double()
        c, ties = (st[:, i].contiguous().view(torch.int32) for i in (3, 4))
        total = e.double().sum(-1)
        above = torch.where(e > bound[:, None], e, 0.).double().sum(-1)
        assert (ties == (e == bound[:, None]).sum(-1)).all()
        assert ((c >= 1) & (c <= ties)).all()
        assert (above < top_p * total * (1 + 1e-5)).all()
        assert (above + c * bound.double() >= top_p * total * (1 - 1e-5)).all()
        assert (above + (c - 1) * bound.double() <= top_p * total * (1 + 1e-5)).all()
        assert ((above + c * bound.double()) / kept - 1).abs().max() < 1e-5
