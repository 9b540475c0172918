"""Algorithm 8 on blocks too tall for one resident column (past 8.7 million rows
on 152 SMs): panels of 16 on W in memory, bit for bit against the oracle's FP32
process, at one panel, one column more, and a ragged third."""
import numpy as np
import pytest

from oracle import ofrr as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


@pytest.mark.parametrize("n,k", [(9000001, 16), (9000001, 17), (8900000, 37)])
def test_tall_blocks_bitexact(rr, n, k):
    W = np.random.default_rng(k).standard_normal((n, k), dtype=np.float32)
    Wd = torch.from_numpy(np.ascontiguousarray(W.T)).cuda().t()
    Q, piv, err = rr.rr_hessenberg(Wd, qtype=torch.float32)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    _, pivo, _, Qo = O.hessenberg(W, arith="f32")
    assert np.array_equal(piv.cpu().numpy(), np.asarray(pivo))
    assert np.array_equal(Q.cpu().numpy(), Qo.astype(np.float32))
