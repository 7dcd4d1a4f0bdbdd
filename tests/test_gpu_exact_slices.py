"""Exact-slice quaternion GEMM (qgemm_emu.cu) on integer matrices, where the
product is known exactly: tile edges (128 x 128 and 128 x 64 tiles), K chunk
and K part remainders, every slice count, the level groups and K ranges a
small product is split over."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ints(rng, rows, cols, bits):
    return rng.integers(-(2 ** bits) + 1, 2 ** bits, size=(4, rows, cols), dtype=np.int64)


def _product(a, b):
    """Hamilton product of int64 planes, exact (|sums| < 2^63)."""
    m = lambda p, q: a[p] @ b[q]  # noqa: E731  (int64 matmul)
    return np.stack([m(0, 0) - m(1, 1) - m(2, 2) - m(3, 3), m(0, 1) + m(1, 0) + m(2, 3) - m(3, 2),
                     m(0, 2) - m(1, 3) + m(2, 0) + m(3, 1), m(0, 3) + m(1, 2) - m(2, 1) + m(3, 0)])


SHAPES = [(1, 1, 1), (3, 17, 5), (64, 48, 80), (60, 512, 60), (128, 64, 128), (129, 65, 127), (300, 1025, 70),
          (60, 768, 200), (257, 130, 385), (70, 2049, 66), (520, 130, 520)]


@pytest.mark.parametrize("m,k,n", SHAPES)
@pytest.mark.parametrize("slices,abits,bbits", [(2, 6, 5), (3, 13, 6), (4, 13, 13), (5, 20, 13), (6, 27, 13),
                                                (7, 27, 20), (8, 27, 13)])
def test_integer_product_is_exact(m, k, n, slices, abits, bbits):
    # abits, bbits: slices 0 .. (bits - 7) / 7 (rounded up) of each operand hold
    # the integers, so every level of the product is formed (sum of the slice
    # indices < slices) and every part of it is a multiple of the fixed-point
    # unit; |sums| < 4 K 2^(abits + bbits) < 2^53 except where noted
    from paper_2605_01464_gb300 import qpinv
    rng = np.random.default_rng(m * 131 + k * 17 + n + slices)
    if abits + bbits + 2 + int(np.ceil(np.log2(k))) > 53:
        abits = 53 - bbits - 2 - int(np.ceil(np.log2(k)))
    a, b = _ints(rng, m, k, abits), _ints(rng, k, n, bbits)
    ctx = qpinv.Context(0)
    c = ctx.qgemm(torch.from_numpy(a.astype(np.float64)).cuda(), torch.from_numpy(b.astype(np.float64)).cuda(),
                  precision="emu", split_level=slices).cpu().numpy()
    ctx.close()
    np.testing.assert_array_equal(c, _product(a, b).astype(np.float64))


@pytest.mark.parametrize("m,k,n", SHAPES)
def test_full_width_product(m, k, n):
    # 40-bit times 21-bit integers use the low levels: the error is the
    # rounding of the eight products' fixed point (unit 2^-F of the operands'
    # scales, F = 62 - ceil(log2 4K), at most two roundings each of up to four
    # parts, and a component takes one product and half of four) plus the
    # dropped levels' 2^-56 K, and the FP64 rounding of the result
    from paper_2605_01464_gb300 import qpinv
    rng = np.random.default_rng(7 * m + k + n)
    a, b = _ints(rng, m, k, 40), _ints(rng, k, n, 21 - max(0, int(np.ceil(np.log2(k))) + 2 - 2))
    ctx = qpinv.Context(0)
    c = ctx.qgemm(torch.from_numpy(a.astype(np.float64)).cuda(), torch.from_numpy(b.astype(np.float64)).cuda(),
                  precision="emu", split_level=8).cpu().numpy()
    ctx.close()
    ref = _product(a, b)
    ea = np.ceil(np.log2(np.abs(a).max(axis=(0, 2)) + 1.0))[:, None]
    eb = np.ceil(np.log2(np.abs(b).max(axis=(0, 1)) + 1.0))[None, :]
    F = 62 - int(np.ceil(np.log2(4 * k)))
    tol = np.exp2(ea + eb) * (3 * 8 * 2.0 ** -F + k * 2.0 ** -55) + np.abs(ref) * 2.0 ** -52
    assert np.all(np.abs(c - ref.astype(np.float64)) <= tol)
