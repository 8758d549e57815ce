"""The junction's backward with its gradients written over o and e, on each of
its three paths: the same bits as with buffers of their own."""
import pytest
import torch

from paper_2608_09703_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,dp,de", [
    (torch.bfloat16, 520, 264),    # register cache
    (torch.float32, 264, 1000),
    (torch.bfloat16, 3080, 1016),  # TMA ring
    (torch.float32, 1540, 2052),
    (torch.bfloat16, 9000, 5544),  # streaming, both segments ending inside a batch of loads
    (torch.float32, 3000, 5192),
])
@pytest.mark.parametrize("embed_first", [False, True])
def test_gradients_over_inputs(dtype, dp, de, embed_first):
    gen = torch.Generator(device="cuda").manual_seed(dp)
    r = lambda n, s: (torch.randn(701, n, generator=gen, device="cuda") * s).to(dtype)
    o, e, g = r(dp, 4.0), r(de, 0.05), r(dp + de, 1.0)
    d_o, d_e = torch.empty_like(o), torch.empty_like(e)
    B.mls_junction_bwd(o, e, g, d_o, d_e, embed_first)
    B.mls_junction_bwd(o, e, g, o, e, embed_first)
    assert torch.equal(o, d_o) and torch.equal(e, d_e)
    assert B.mls_get_status() == 0
