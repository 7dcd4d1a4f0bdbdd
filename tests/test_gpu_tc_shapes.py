"""The tensor-core GEMM's tile shapes and fused epilogue at tile edges: the
shapes chosen by size (qpinv_options.tc_broad = -1, 0, 1) give bit-identical
products, and fused combine passes the same iterates as the separate kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_01464_gb300 import qpinv
    c = qpinv.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (15, 33, 17), (16, 32, 16), (31, 70, 65), (127, 31, 33), (128, 96, 128),
                                   (129, 65, 31), (200, 300, 257), (1000, 64, 16)])
@pytest.mark.parametrize("split", [1, 2, 3])
def test_shapes_give_the_same_bits(ctx, m, k, n, split):
    g = torch.Generator(device="cuda").manual_seed(m + 7 * k + 31 * n)
    a = torch.randn(4, m, k, generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn(4, k, n, generator=g, device="cuda", dtype=torch.float64)
    out = []
    for broad in ("auto", False, True):
        ctx.configure(tc_broad=broad)
        out.append(ctx.qgemm(a, b, precision="tc", split_level=split).cpu().numpy())
    ctx.configure(tc_broad="auto")
    np.testing.assert_array_equal(out[1], out[0])
    np.testing.assert_array_equal(out[2], out[0])
    # BF16 terms carry 8 bits each; FP32 accumulation adds about 2^-23 per K step of 4 K terms
    ref = torch.stack([a[0] @ b[0] - a[1] @ b[1] - a[2] @ b[2] - a[3] @ b[3],
                       a[0] @ b[1] + a[1] @ b[0] + a[2] @ b[3] - a[3] @ b[2],
                       a[0] @ b[2] - a[1] @ b[3] + a[2] @ b[0] + a[3] @ b[1],
                       a[0] @ b[3] + a[1] @ b[2] - a[2] @ b[1] + a[3] @ b[0]]).cpu().numpy()
    scale = np.linalg.norm(a.cpu().numpy(), axis=(0, 2))[:, None] * np.linalg.norm(b.cpu().numpy(), axis=(0, 1))[None]
    assert np.all(np.abs(out[0] - ref) <= (3 * 2.0 ** (-8 * split) + 4 * k * 2.0 ** -22) * scale)


@pytest.mark.parametrize("m,n", [(17, 17), (33, 31), (64, 64), (65, 129), (130, 97), (257, 257)])
@pytest.mark.parametrize("method", ["qhpi19", "qsai", "qrapid"])
def test_fused_epilogue_matches_the_separate_pass(ctx, m, n, method):
    # the same element arithmetic in both; only the FP32 sums of the stop test
    # group differently, so the iterates agree to rounding of the last steps
    g = torch.Generator(device="cuda").manual_seed(m * n)
    a = torch.randn(4, m, n, generator=g, device="cuda", dtype=torch.float64)
    xs = []
    for fuse in (True, False):
        ctx.configure(fuse_epilogue=fuse)
        x, info = ctx.solve(a, method, tol=1e-12)
        assert info["status"] in ("converged", "plateau")
        xs.append(x.cpu().numpy())
    ctx.configure(fuse_epilogue=True)
    assert np.linalg.norm(xs[0] - xs[1]) <= 1e-10 * np.linalg.norm(xs[1])


@pytest.mark.parametrize("m,k,n", [(2, 1, 7), (130, 1, 150), (1300, 1100, 1150)])
@pytest.mark.parametrize("broad", ["auto", False, True])
def test_fp64_output_of_special_values(ctx, m, k, n, broad):
    # column 0 of A times row 0 of B, all others zero: every entry of plane 0 is
    # one exact FP32 product (zero, normal, largest, smallest, infinite, NaN)
    va = torch.tensor([1.0, 0.0, -3.0, 2.0 ** 100, -2.0 ** -100, 1.9921875 * 2.0 ** 127, float("inf"), float("nan")],
                      dtype=torch.float64, device="cuda")
    vb = torch.tensor([1.0, -0.5, 2.0 ** -20, 2.0 ** 20, 0.0], dtype=torch.float64, device="cuda")
    a = torch.zeros(4, m, k, dtype=torch.float64, device="cuda")
    b = torch.zeros(4, k, n, dtype=torch.float64, device="cuda")
    a[0, :, 0] = va[torch.arange(m, device="cuda") % 8]
    b[0, 0, :] = vb[torch.arange(n, device="cuda") % 5]
    ctx.configure(tc_broad=broad)
    c = ctx.qgemm(a, b, precision="tc", split_level=1)
    ctx.configure(tc_broad="auto")
    e = torch.zeros_like(c)
    for q in range(4):  # 0 x inf and 0 x NaN of the zero planes are NaN
        e[q] = (a[0, :, :1] * b[q, :1, :]).float().double()
    ok = (c == e) | (torch.isnan(c) & torch.isnan(e))
    # a product below FP32's normal range may come out as zero
    ok |= (e.abs() < 2.0 ** -126) & (c.abs() < 2.0 ** -126)
    # one K step adds zeros to an infinity: nothing but it or NaN can come out
    if k > 1:
        ok |= ~torch.isfinite(a[0, :, :1]).expand(m, n) & ~torch.isfinite(c[0])
    assert bool(ok.all())


@pytest.mark.parametrize("m,k,n", [(700, 90, 650), (1153, 33, 705)])
def test_clustered_shapes_give_the_same_bits(ctx, m, k, n):
    # enough items that the 64-column shape runs in clusters, odd tile counts
    test_shapes_give_the_same_bits(ctx, m, k, n, 2)
