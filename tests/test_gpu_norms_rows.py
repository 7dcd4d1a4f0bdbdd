"""Norms of matrices with more rows than 65535 blocks of 64, through the
features of the learned alpha (||A||_F, ||A||_1, ||A||_inf among them)."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(64 * 65535, 1), (64 * 65535 + 1, 1), (64 * 65540 + 3, 33), (3, 32 * 65535 + 1)])
def test_norms_of_long_matrices(m, n):
    from paper_2605_01464_gb300 import qpinv
    g = torch.Generator(device="cuda").manual_seed(m + n)
    a = torch.randn(4, m, n, generator=g, device="cuda", dtype=torch.float64)
    ctx = qpinv.Context(0)
    feat, theta1 = ctx.alpha_features(a)
    ctx.close()
    mod = a.square().sum(0).sqrt()
    # logarithms as FP32 numbers (below 32 in modulus: half an ulp is 2^-20)
    for i, x in ((3, a.norm().item()), (4, mod.sum(0).max().item()), (5, mod.sum(1).max().item())):
        assert abs(float(feat[i]) - math.log(x)) <= 2.0 ** -19, i
    # the Ritz value is below ||A||_F^2, and for one column equals it
    assert theta1 <= a.square().sum().item() * (1 + 1e-5)
    if n == 1:
        assert theta1 >= a.square().sum().item() * (1 - 1e-5)
