"""FP64 products with more rows than one grid takes (524280 per launch): just
over one launch's, and as many as the interface can name, where a 32-bit row
counter would step past the largest int."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [524281, 2 ** 31 - 1])
def test_rows_in_slabs(m):
    from paper_2605_01464_gb300 import qpinv
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 80 * m:
        pytest.skip("needs %d GB of device memory" % (80 * m >> 30))
    a = torch.arange(m, dtype=torch.float64, device="cuda")
    b = torch.tensor([1.0, 2.0, -1.0, 3.0], dtype=torch.float64, device="cuda").view(4, 1, 1)
    c = torch.full((4, m, 1), float("nan"), dtype=torch.float64, device="cuda")
    ctx = qpinv.Context(0)
    # four equal planes, one in memory: (a, a, a, a) (1, 2, -1, 3), exact integers
    ctx.qgemm(a.view(1, m, 1).expand(4, m, 1), b, precision="fp64", C=c)
    ctx.close()
    for plane, x in enumerate((1 - 2 + 1 - 3, 2 + 1 + 3 + 1, -1 - 3 + 1 + 2, 3 - 1 - 2 + 1)):
        assert torch.equal(c[plane, :, 0], a * x), plane
    del a, c
    torch.cuda.empty_cache()
