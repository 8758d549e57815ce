"""The junction's register cache with every pair of vectors per lane (1, 2, 4, 8)
that the two segments can take, one of them ending inside its last vector."""
import pytest
import torch

from test_junction import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,unit", [(torch.bfloat16, 8), (torch.float32, 4)])
@pytest.mark.parametrize("ro", [1, 2, 4, 8])
@pytest.mark.parametrize("re", [1, 2, 4, 8])
def test_segment_vectors(dtype, unit, ro, re):
    """Tolerances as in test_junction.py: one rounding to the storage type, or
    fp32 sums of at most 2048 terms."""
    g = torch.Generator().manual_seed(100 * ro + re)
    T, dp, de = 9, (32 * ro - 3) * unit, 32 * re * unit
    o = (torch.randn(T, dp, generator=g) * 3).to(dtype)
    e = (torch.randn(T, de, generator=g) * 0.1).to(dtype)
    gr = torch.randn(T, dp + de, generator=g).to(dtype)
    o[5] = 0
    bf = dtype == torch.bfloat16
    for embed_first in (False, True):
        compare(o, e, gr, embed_first, tol_x=4e-3 if bf else 1e-5, tol_g=1e-2 if bf else 1e-5)
