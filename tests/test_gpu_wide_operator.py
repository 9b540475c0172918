"""FP64-accurate products with operators of very many columns (the grids of the
exponent passes run over columns): A^T Y past 65535 columns, A X past 65535
groups of 128 columns.  Small integers, whose sums are exact in FP64."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


def ints(rows, cols, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-8, 9, (cols, rows), generator=g, device="cuda").double().t()


@pytest.mark.parametrize("trans,m,n,N", [(1, 16, 65536, 3), (1, 8, 70008, 17), (0, 8, 65536 * 128 + 8, 1)])
@pytest.mark.parametrize("slices", [8, 10])
def test_products_of_wide_operators(rr, trans, m, n, N, slices):
    A, X = ints(m, n, 1), ints(m if trans else n, N, 2)
    C = rr.rr_gemm_f64_emulated(trans, A, X, slices=slices)
    assert torch.equal(C, (A.t() if trans else A) @ X)
