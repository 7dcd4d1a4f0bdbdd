"""Exact-slice products and solves with little device memory left: the slices
of all eight products of an operand take twice the memory of the four-plane
form, so a call that does not get them works in two groups of four, gives back
what it holds of the wide form, and returns the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# allocations come in 2 MB pages, ten or so buffers in each call, and the driver
# keeps some memory to itself
SLACK = 32 << 20


def _randn(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _limited(call, out, options, saved):
    """`call` writes `out`: with ample memory, then twice on a new context with
    `saved` bytes less free memory than its workspace took."""
    from paper_2605_01464_gb300 import qpinv
    c = qpinv.Context(0, **options)
    call(c)  # also loads every kernel
    c.close()
    want, got = out.clone(), [torch.empty_like(out), torch.empty_like(out)]
    for x in got:
        x.copy_(torch.zeros_like(out).zero_())
    f0 = _free()
    c = qpinv.Context(0, **options)
    call(c)
    used = f0 - _free()
    c.close()
    ballast = torch.empty(_free() - used + saved, dtype=torch.uint8, device="cuda")
    try:
        c = qpinv.Context(0, **options)
        for x in got:
            out.zero_()
            call(c)
            x.copy_(out)
        c.close()
    finally:
        del ballast
        torch.cuda.empty_cache()
    for x in got:
        assert torch.equal(x, want)


@pytest.mark.parametrize("slices", [6, 8])
def test_product(slices):
    # two operands' slices: 8 products x S slices x 2 bytes per entry each; half of
    # both is to be saved
    m, k, n = 1000, 1500, 1200
    a, b = _randn(1, 4, m, k), _randn(2, 4, k, n)
    out = torch.empty(4, m, n, dtype=torch.float64, device="cuda")
    ld = (k + 63) // 64 * 64
    saved = 8 * slices * (m + n) * ld - SLACK

    _limited(lambda c: c.qgemm(a, b, precision="emu", split_level=slices, C=out), out, {}, saved)


@pytest.mark.parametrize("precision,method,m,n", [("emu", "qsai", 768, 768), ("emu", "ns", 1000, 700),
                                                  ("mixed", "qhpi19", 768, 768), ("mixed", "qsai", 700, 1000)])
def test_solve(precision, method, m, n):
    # at least the residual product's two operands (one of them A, kept) and one
    # more operand's slices are held at once: half of three matrices' slices
    a = _randn(m + n, 4, m, n)
    x = torch.empty(4, n, m, dtype=torch.float64, device="cuda")
    saved = 3 * 64 * m * n - SLACK

    _limited(lambda c: c.solve(a, method, tol=1e-12, X=x), x, dict(precision=precision), saved)
