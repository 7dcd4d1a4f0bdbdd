"""Products and solves on the caller's own planes: leading dimensions above the
width, bases off the 16-byte boundary, planes interleaved by rows, in reverse
order and at irregular distances, and results that share memory with an
operand.  Every call must give the bits of the same call on contiguous copies
and leave the entries around a result's rows alone."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_01464_gb300 import qpinv
    c = qpinv.Context(0)
    yield c
    c.close()


FORMS = ["ld", "odd", "interleaved", "shared"]


def _view(form, rows, cols):
    """A (4, rows, cols) view of NaN-filled memory, and that memory."""
    if form == "ld":
        buf = torch.full((4, rows + 2, cols + 6), float("nan"), dtype=torch.float64, device="cuda")
        return buf[:, 1:rows + 1, 4:cols + 4], buf
    if form == "odd":
        buf = torch.full((4 * (rows + 1) * (cols + 3) + 4,), float("nan"), dtype=torch.float64, device="cuda")
        ld = cols + 2 + (cols + 1) % 2  # odd
        return buf.as_strided((4, rows, cols), (rows * ld, ld, 1), 1), buf
    if form == "interleaved":  # row i of the four planes side by side
        buf = torch.full((rows, 4, cols), float("nan"), dtype=torch.float64, device="cuda")
        return buf.permute(1, 0, 2), buf
    buf = torch.full((4, rows, cols), float("nan"), dtype=torch.float64, device="cuda")
    return buf, buf


def _fill(form, x):
    v, buf = _view(form, x.shape[1], x.shape[2])
    v.copy_(x)
    return v, buf


def _randn(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


PRECISIONS = [("tc", 1), ("tc", 3), ("emu", 4), ("emu", 8), ("fp64", 1)]


@pytest.mark.parametrize("precision,split", PRECISIONS)
@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (33, 20, 17), (130, 71, 65)])
@pytest.mark.parametrize("form", FORMS)
def test_product_on_views(ctx, precision, split, m, k, n, form):
    a, b = _randn(m + k, 4, m, k), _randn(k + n + 1, 4, k, n)
    want = ctx.qgemm(a, b, precision=precision, split_level=split)
    va, _ = _fill(form, a)
    vb, _ = _fill(form, b)
    vc, buf = _view(form, m, n)
    ctx.qgemm(va, vb, precision=precision, split_level=split, C=vc)
    assert torch.equal(vc, want)
    vc.fill_(float("nan"))  # what is left was never part of the result
    assert bool(torch.isnan(buf).all())


@pytest.mark.parametrize("precision,split", PRECISIONS)
@pytest.mark.parametrize("other", ["a", "b"])
def test_result_over_an_operand(ctx, precision, split, other):
    n = 70
    a, b = _randn(3, 4, n, n), _randn(4, 4, n, n)
    want = ctx.qgemm(a, b, precision=precision, split_level=split)
    big = torch.zeros(4, n + 1, n, dtype=torch.float64, device="cuda")
    x = big[:, :n]
    x.copy_(a if other == "a" else b)
    c = big[:, 1:]  # one row further down than the operand
    ctx.qgemm(x if other == "a" else a, x if other == "b" else b, precision=precision, split_level=split, C=c)
    assert torch.equal(c, want)


@pytest.mark.parametrize("precision,split", PRECISIONS)
def test_reversed_and_irregular_planes(ctx, precision, split):
    # through the C interface: four separate plane pointers
    from paper_2605_01464_gb300 import qpinv
    m, k, n = 40, 33, 21
    a, b = _randn(5, 4, m, k), _randn(6, 4, k, n)
    want = ctx.qgemm(a, b, precision=precision, split_level=split)
    ra = a.flip(0).contiguous()  # plane t at position 3 - t: a negative distance
    parts = [_randn(7 + t, k * n + 13 * t + 1) for t in range(4)]  # irregular distances
    for t in range(4):
        parts[t][:k * n].view(k, n).copy_(b[t])
    rc = torch.empty(4, m, n, dtype=torch.float64, device="cuda")
    pa = qpinv.PTR4(*[ra[3 - t].data_ptr() for t in range(4)])
    pb = qpinv.PTR4(*[parts[t].data_ptr() for t in range(4)])
    pc = qpinv.PTR4(*[rc[3 - t].data_ptr() for t in range(4)])
    prec = {"tc": 2, "emu": 3, "fp64": 0}[precision]
    torch.cuda.synchronize()
    assert qpinv.lib().qpinv_qgemm(ctx.h, ctypes.c_void_p(0), m, k, n, pa, k, pb, n, pc, n, prec, split) == 0
    assert torch.equal(rc.flip(0), want)


@pytest.mark.parametrize("precision", ["mixed", "emu", "fp64"])
@pytest.mark.parametrize("m,n", [(40, 33), (33, 40), (65, 65)])
@pytest.mark.parametrize("form", FORMS)
def test_solve_on_views(ctx, precision, m, n, form):
    a = _randn(m * n, 4, m, n)
    ctx.configure(precision=precision)
    want, winfo = ctx.solve(a, "qsai", tol=1e-12)
    va, abuf = _fill(form, a)
    before = abuf.clone()
    vx, xbuf = _view(form, n, m)
    x, info = ctx.solve(va, "qsai", tol=1e-12, X=vx)
    ctx.configure(precision="mixed")
    assert torch.equal(vx, want) and info["iters"] == winfo["iters"] and info["E"] == winfo["E"]
    assert torch.equal(torch.nan_to_num(abuf), torch.nan_to_num(before))
    vx.fill_(float("nan"))
    assert bool(torch.isnan(xbuf).all())


@pytest.mark.parametrize("n", [64, 65])
def test_pseudoinverse_over_its_matrix(ctx, n):
    a = _randn(n, 4, n, n)
    want, winfo = ctx.solve(a, "qhpi19", tol=1e-12)
    x, info = ctx.solve(a, "qhpi19", tol=1e-12, X=a)
    assert torch.equal(a, want) and info["E"] == winfo["E"]
