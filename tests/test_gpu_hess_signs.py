"""The blocked process keeps the sign of a zero: a panel of r columns updates its
trailing columns with its own r products and no padding, so W and Q equal the
unblocked process's in every bit, zeros' signs included."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


@pytest.mark.parametrize("panel", [1, 5, 8, 13, 16, 31, 32])
def test_blocked_process_keeps_signed_zeros(rr, panel):
    # pivots on the diagonal; in the rows below, zeros whose sign every step
    # keeps: -0 - (w * +0) with w > 0 by the first panel's columns, -0 - (w * -0)
    # with w < 0 by the later ones
    n, k = 1000, panel + 7
    W = np.zeros((n, k), dtype=np.float32)
    W[:, panel:] = -0.0
    for j in range(k):
        W[j, j] = 4.0
        W[j, j + 1:] = 1.0 if j < panel else -1.0
    out = []
    for f in (lambda w: rr.rr_hessenberg(w, qtype=torch.float32),
              lambda w: rr.rr_hessenberg_blocked(w, qtype=torch.float32, panel=panel)):
        Wd = torch.from_numpy(np.ascontiguousarray(W.T)).cuda().t()
        Q, piv = f(Wd)[:2]
        out.append((Wd.t().contiguous().view(torch.int32), Q.t().contiguous().view(torch.int32), piv))
    torch.cuda.synchronize()
    assert bool(torch.signbit(out[0][0].view(torch.float32)[panel:, k:]).all())
    for a, b in zip(*out):
        assert torch.equal(a, b)
