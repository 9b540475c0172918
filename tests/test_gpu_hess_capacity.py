"""Algorithm 8 at the edge of what the CTAs' shared memory holds: blocks whose
slab fills a CTA of the one-cluster form (216 and more columns on up to 16
CTAs), and their neighbours one row or column further on either side (the
cluster, the cooperative grid, panels of 32), bit for bit against the oracle's
FP32 process."""
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


@pytest.mark.parametrize("n,k", [(246, 224), (247, 224), (248, 224), (427, 256), (428, 256), (429, 256), (988, 224),
                                 (1024, 215), (1024, 216), (607, 512), (608, 512), (3424, 256), (3968, 223),
                                 (4096, 216), (4097, 216), (4096, 217)])
def test_shared_memory_edge_bitexact(rr, n, k):
    W = np.random.default_rng(n + k).standard_normal((n, k)).astype(np.float32)
    _, piv, _, Qf = O.hessenberg(W, arith="f32")
    Wd = torch.from_numpy(np.ascontiguousarray(W.T)).cuda().t()
    Q, p, err = rr.rr_hessenberg(Wd, qtype=torch.float32)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert np.array_equal(p.cpu().numpy(), np.asarray(piv))
    assert np.array_equal(Q.cpu().numpy(), Qf.astype(np.float32)) and np.array_equal(Wd.cpu().numpy(), Q.cpu().numpy())
