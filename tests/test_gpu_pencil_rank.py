"""Pencils with more than 32 singular values together: far more columns than rows
(the others are zeros), low rank, columns graded over many decades, and a large
group of equal or close values.  Values and vectors outside the group are as
accurate as in any other pencil, and the group stays finite and near its values."""
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


def _randn(*shape, seed):
    return torch.randn(*shape, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


def _check(rr, B, k):
    """B's pencil with unit Grams: the first k values and vectors as in any pencil (64 n eps, as
    FP64 products of length n in whitening, four refinement steps and read-out add up), the other
    values within the FP32 Jacobi's floor (column norms count as converged below 1e-5 of the largest)."""
    b1, b2 = B.shape
    eye = lambda n: rr.fortran(torch.eye(n, dtype=torch.float64, device="cuda"))  # noqa: E731
    s, Y, Z, _ = rr.rr_pencil_svd(rr.fortran(B.cuda()), eye(b1), eye(b2))
    ref = torch.linalg.svdvals(B)
    s, Y, Z = s.cpu(), Y[:, :k].cpu(), Z[:, :k].cpu()
    tol = 64 * max(b1, b2) * EPS
    smax = float(ref[0])
    assert float((s[:k] - ref[:k]).abs().max()) <= tol * smax
    assert float((s[k:] - ref[k:]).abs().max() if k < len(ref) else 0.0) <= 1e-5 * max(b1, b2) ** 0.5 * smax
    one = torch.eye(k, dtype=torch.float64)
    grow = smax / torch.minimum(ref[:k, None], ref[None, :k])
    for W in (Y, Z):
        assert bool(((W.t() @ W - one).abs() <= tol * grow).all())
    assert bool(((Y.t() @ B @ Z - torch.diag(ref[:k])).abs() <= tol * smax * grow).all())


@pytest.mark.parametrize("b1,b2", [(1, 200), (17, 335), (36, 68), (36, 72), (36, 100), (100, 200), (200, 255)])
def test_many_more_columns_than_rows(rr, b1, b2):
    _check(rr, _randn(b1, b2, seed=b1 + b2), b1)


@pytest.mark.parametrize("b1,b2,rank", [(64, 64, 20), (100, 100, 20), (256, 256, 100), (320, 320, 40), (300, 200, 100)])
def test_low_rank(rr, b1, b2, rank):
    _check(rr, _randn(b1, rank, seed=b1) @ _randn(rank, b2, seed=rank), rank)


@pytest.mark.parametrize("b,decades", [(130, 9), (200, 8), (256, 9), (320, 7), (320, 12)])
def test_graded_columns(rr, b, decades):
    B = _randn(b, b, seed=b) * torch.logspace(0, -decades, b, dtype=torch.float64)
    s = torch.linalg.svdvals(B)
    _check(rr, B, int((s > 1e-4 * s[0]).sum()))


@pytest.mark.parametrize("b,decades", [(96, 9), (130, 8), (200, 7), (240, 7), (256, 6)])
def test_graded_columns_that_separate(rr, b, decades):
    """Small groups and mild angles across their cuts: every value and vector as accurate as any."""
    _check(rr, _randn(b, b, seed=b) * torch.logspace(0, -decades, b, dtype=torch.float64), b)


@pytest.mark.parametrize("spread", [0.0, 1e-8, 1e-5])
def test_sixty_close_values(rr, spread):
    """60 of 120 values within `spread`: finite, orthonormal to 1e-5, values within the Jacobi's
    1e-4 relative orthogonality of a group of 60 (Gershgorin: 60 1e-4 / 2 of the value)."""
    b = 120
    Q, P = (torch.linalg.qr(_randn(b, b, seed=i))[0] for i in (1, 2))
    ref = torch.cat([1 + spread * torch.linspace(1, 0, 60, dtype=torch.float64),
                     torch.linspace(0.9, 0.1, 60, dtype=torch.float64)])
    eye = rr.fortran(torch.eye(b, dtype=torch.float64, device="cuda"))
    s, Y, Z, _ = rr.rr_pencil_svd(rr.fortran(((Q * ref) @ P.t()).cuda()), eye, eye)
    s, Y, Z = s.cpu(), Y.cpu(), Z.cpu()
    assert float((s[:60] - ref[:60]).abs().max()) <= 60 * 1e-4 / 2
    tol = 64 * b * EPS
    assert float((s[60:] - ref[60:]).abs().max()) <= tol
    one = torch.eye(b, dtype=torch.float64)
    assert float((Z.t() @ Z - one).abs().max()) <= 1e-5
    for W in (Y, Z):
        assert float((W.t() @ W - one)[60:, 60:].abs().max()) <= 10 * tol
