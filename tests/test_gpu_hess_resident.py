"""Algorithm 8 with the block resident in the CTAs' shared memory (panels of 8
columns), bit for bit against the oracle's FP32 process: one to several panels,
ragged panels and row counts, more CTAs than one polling warp covers, ties and
skipped columns at panel edges, padded leading dimensions, and blocks whose
columns fit only in part (several launches per panel of 32)."""
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


def run(rr, W, qtype, ld=None):
    n, k = W.shape
    buf = torch.zeros(k, ld or n, dtype=torch.float32, device="cuda")
    buf[:, :n] = torch.from_numpy(np.ascontiguousarray(W.T)).cuda()
    Wd = buf.t()[:n]
    Q, piv, err = rr.rr_hessenberg(Wd, qtype=qtype)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    return Wd.cpu().numpy(), Q.float().cpu().numpy(), piv.cpu().numpy()


@pytest.mark.parametrize("n,k,ld", [(1, 1, None), (9, 8, None), (127, 9, 130), (129, 16, None), (1000, 33, 1001),
                                    (4097, 24, None), (20001, 41, None), (60000, 17, 60003)])
def test_resident_bitexact(rr, n, k, ld):
    W = np.random.default_rng(n + k).standard_normal((n, k)).astype(np.float32)
    _, piv, _, Qf = O.hessenberg(W, arith="f32")
    Wd, Q, p = run(rr, W, torch.float32, ld)
    assert np.array_equal(p, np.asarray(piv))
    assert np.array_equal(Q, Qf.astype(np.float32)) and np.array_equal(Wd, Q)


def test_resident_ties_and_skips_at_panel_edges(rr):
    rng = np.random.default_rng(8)
    W = rng.integers(-3, 4, (3000, 40)).astype(np.float32)     # many ties
    W[:, 7] = W[:, 3]                                          # last of a panel
    W[:, 8] = W[:, 0] - W[:, 2]                                # first of the next
    W[:, 16:24] = 0                                            # a whole panel
    _, piv, _, Qf = O.hessenberg(W, arith="f32")
    _, Q, p = run(rr, W, torch.bfloat16)
    assert np.array_equal(p, np.asarray(piv))
    assert np.array_equal(Q, O.round_bf16(Qf).astype(np.float32))


@pytest.mark.parametrize("n,k", [(600000, 37), (1100001, 12)])
def test_columns_resident_in_part(rr, n, k):
    rng = np.random.default_rng(n)
    W = rng.standard_normal((n, k)).astype(np.float32)
    _, piv, _, Qf = O.hessenberg(W, arith="f32")
    Wd, Q, p = run(rr, W, torch.float32)
    assert np.array_equal(p, np.asarray(piv))
    assert np.array_equal(Q, Qf.astype(np.float32)) and np.array_equal(Wd, Q)
