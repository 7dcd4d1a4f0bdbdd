"""Exact-slice products at the largest value their fixed point has to hold:
every entry of A's rows and B's columns just below its power of two, all four
components of equal modulus, signs such that one component of the product
collects them all (4 K of the operands' scales; the combine pass forms twice
that).  Slices that cannot hold the whole mantissa round such entries up to the
power of two itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the right factor's signs that put the maximum into w, x, y and z for a left
# factor (1, 1, 1, 1)
SIGNS = [(1, -1, -1, -1), (1, 1, -1, 1), (1, 1, 1, -1), (1, -1, 1, 1)]


def _hamilton(p, q):
    return [p[0] * q[0] - p[1] * q[1] - p[2] * q[2] - p[3] * q[3],
            p[0] * q[1] + p[1] * q[0] + p[2] * q[3] - p[3] * q[2],
            p[0] * q[2] - p[1] * q[3] + p[2] * q[0] + p[3] * q[1],
            p[0] * q[3] + p[1] * q[2] - p[2] * q[1] + p[3] * q[0]]


@pytest.mark.parametrize("slices", range(2, 9))
@pytest.mark.parametrize("k", [1, 2, 5, 64, 128])
@pytest.mark.parametrize("below", [2.0 ** -53, 2.0 ** -45])
def test_largest_component(slices, k, below):
    from paper_2605_01464_gb300 import qpinv
    v = 1.0 - below
    m, n = 3, 5
    # The operands' exponents are 0.  A slicing rounds an entry by at most half of
    # 2^-7S (each factor's, times a factor below 1: 2^-7S per product of entries);
    # the dropped levels hold the S - 1 digit pairs of level S, below 2^12
    # 2^-7(S+2) each, and geometrically less: S 2^-7S / 4 bounds them.  4 K
    # products of entries.  Fixed point: unit 2^-F, F >= 61 - ceil(log2 4K), a
    # few roundings in each of five products.  The result's own rounding: 2^-53.
    lg = int(np.ceil(np.log2(4 * k)))
    tol = 4 * k * ((1.0 + slices / 4.0) * 2.0 ** (-7 * slices) * 1.01 + 2.0 ** -52) + 24 * 2.0 ** (lg - 61)
    ctx = qpinv.Context(0)
    for signs in SIGNS:
        for neg in (1.0, -1.0):
            a = torch.full((4, m, k), v, dtype=torch.float64, device="cuda")
            b = torch.full((4, k, n), v, dtype=torch.float64, device="cuda")
            b *= neg * torch.tensor(signs, dtype=torch.float64, device="cuda")[:, None, None]
            c = ctx.qgemm(a, b, precision="emu", split_level=slices).cpu().numpy()
            ref = neg * k * v * v * np.array(_hamilton((1, 1, 1, 1), signs), dtype=np.float64)
            assert np.abs(ref).max() > 3.9 * k
            assert np.all(np.abs(c - ref[:, None, None]) <= tol), (signs, neg, c[:, 0, 0], ref)
    ctx.close()
