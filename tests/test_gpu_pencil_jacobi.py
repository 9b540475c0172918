"""Block Jacobi rounds on the block's Gram matrix, through the pencil solvers:
sizes at the edges of the column blocks (one column, odd widths, partly filled
groups of 4 and 8 columns and of 4 rows, one CTA to a full cluster, the wide
form past it), columns whose norms span nine decades, and nothing to rotate.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


def _check(rr, B):
    b1, b2 = B.shape
    nn = min(b1, b2)
    cm = lambda t: t.t().contiguous().t()  # noqa: E731  (column-major, as the library takes its blocks)
    eye = lambda n: cm(torch.eye(n, dtype=torch.float64, device="cuda"))  # noqa: E731
    s, Y, Z, _ = rr.rr_pencil_svd(cm(B), eye(b1), eye(b2))
    n = max(b1, b2)
    ref = torch.linalg.svdvals(B.cpu()).cuda()
    smax = float(ref[0])
    # FP64 products of length n in whitening, refinement (V <- V (I + E), four
    # times) and read-out: a few n eps each, taken together as 64 n eps of the
    # largest value; a left vector is C v / sigma, so it carries that error over
    # its own value
    tol = 64 * n * EPS
    assert float((s[:nn] - ref).abs().max()) <= tol * smax
    grow = smax / torch.minimum(ref[:, None], ref[None, :])
    for W in (Y[:, :nn], Z[:, :nn]):
        D = (W.t() @ W - torch.eye(nn, dtype=torch.float64, device="cuda")).abs()
        assert bool((D <= tol * grow).all())
    R = (Y[:, :nn].t() @ B @ Z[:, :nn] - torch.diag(ref)).abs()
    assert bool((R <= tol * smax * grow).all())


@pytest.mark.parametrize("b1,b2", [(1, 1), (2, 3), (5, 9), (17, 33), (36, 64), (70, 66), (131, 131), (254, 255),
                                   (257, 260), (300, 290), (300, 250), (200, 170)])
def test_pencil_svd_block_edges(rr, b1, b2):
    g = torch.Generator().manual_seed(100 * b1 + b2)
    _check(rr, torch.randn(b1, b2, generator=g, dtype=torch.float64).cuda())


@pytest.mark.parametrize("b", [24, 64])
def test_pencil_svd_graded_columns(rr, b):
    g = torch.Generator().manual_seed(b)
    B = torch.randn(b, b, generator=g, dtype=torch.float64)
    _check(rr, (B * torch.logspace(0, -9, b, dtype=torch.float64)).cuda())


@pytest.mark.parametrize("b", [4, 65])
def test_pencil_svd_nothing_to_rotate(rr, b):
    _check(rr, torch.diag(torch.linspace(2, 1, b, dtype=torch.float64)).cuda())


@pytest.mark.parametrize("b", [1, 31, 32, 33, 65, 96, 255, 256])
def test_pencil_eig_whitening_tile_edges(rr, b):
    """The Cholesky-inverse's 32 x 32 tiles at their edges: Y^T G Y = I and
    H Y = G Y theta for a Gram matrix of condition below 64."""
    g = torch.Generator().manual_seed(b)
    X = torch.randn(2 * b + 8, b, generator=g, dtype=torch.float64)
    G = X.t() @ X / (2 * b + 8)
    S = torch.randn(b, b, generator=g, dtype=torch.float64)
    H = (S + S.t()) / 2
    w = torch.linalg.eigvalsh(G)
    assert float(w[-1] / w[0]) < 64
    cm = lambda t: t.cuda().t().contiguous().t()  # noqa: E731
    theta, Y, dropped = rr.rr_pencil_eig(cm(H), cm(G))
    assert dropped == 0
    theta, Y = theta.cpu(), Y.cpu()
    # products of length b (64 b eps, as above) times the condition of G
    tol = 64 * 64 * b * EPS
    assert float((Y.t() @ G @ Y - torch.eye(b, dtype=torch.float64)).abs().max()) <= tol
    scale = float(H.abs().sum(0).max()) * float(Y.abs().max())
    assert float((H @ Y - G @ Y * theta).abs().max()) <= tol * max(1.0, scale)
