"""Grams of a Y with more columns than one launch takes: column chunks of 4096 on
the tensor cores, exact on small integers, added to G when asked, and with the
tensor-core path's answer to an infinity (its row NaN) in every chunk."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


@pytest.mark.parametrize("n,p,q,t", [(64, 3, 4096, torch.float64), (72, 5, 4097, torch.bfloat16),
                                     (1000, 40, 9000, torch.float32)])
def test_wide_y_in_chunks(rr, n, p, q, t):
    g = torch.Generator(device="cuda").manual_seed(q)
    X = torch.randint(-8, 9, (p, n), generator=g, device="cuda").double().t()
    Y = torch.randint(-8, 9, (q, n), generator=g, device="cuda").to(t).t()
    ref = X.t() @ Y.double()
    G = rr.rr_gram(X, Y)
    assert torch.equal(G, ref)
    rr.rr_gram(X, Y, G=G, accumulate=True)
    assert torch.equal(G, 2 * ref)
    X[7, 1] = float("inf")
    G = rr.rr_gram(X, Y)
    assert bool(torch.isnan(G[1]).all()) and torch.equal(G[0], ref[0]) and torch.equal(G[2:], ref[2:])
