"""Sampling with a NaN in the verifier's head: the rows have no nucleus, so every
token that is a number is kept and the NaN one never sampled, at every size and
by either logits kernel."""
import pytest
import torch

from paper_2608_09703_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("b,V", [(3, 300), (3, 1003), (3, 20011), (200, 1003), (200, 20011)])
def test_nan_logit_is_never_sampled(b, V, dtype):
    gen = torch.Generator(device="cuda").manual_seed(V)
    H = torch.randn(b, 136, generator=gen, device="cuda").to(dtype)
    W = (torch.randn(V, 136, generator=gen, device="cuda") * 0.2).to(dtype)
    u = torch.rand(b, 1, 2, generator=gen, device="cuda")
    W[5, 3] = float("nan")

    def sample(top_p):
        op = B.SpecVerify(b, 0, V, 64, 136, temperature=0.7, top_p=top_p, dtype=dtype)
        none = torch.empty(b, 0, dtype=torch.int32, device="cuda")
        return op(H[:0, :64].contiguous(), W[:, :64].contiguous(), H, W, none, u)[1].clone()

    got = sample(0.9)
    z = (H.double() @ W.double().T / 0.7).nan_to_num(nan=float("-inf"))
    p = torch.softmax(z, -1)
    cum, want = p.cumsum(-1), u[:, 0, 1, None].double()
    i = got.long()[:, None]
    # the smallest token whose cumulative passes u: to the rounding of p, 2e-3 for tf32 logits
    assert (cum.gather(1, i) > want - 2e-3).all()
    assert (cum.gather(1, i) - p.gather(1, i) < want + 2e-3).all()
    assert (got != 5).all() and torch.equal(got, sample(1.0))
    assert B.mls_get_status() == 0
