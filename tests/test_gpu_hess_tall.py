"""Algorithm 8 on blocks too tall for one resident column (past 8.7 million rows
on 152 SMs): panels of 16 on W in memory, bit for bit against the oracle's FP32
process, at one panel, one column more, and a ragged third.  (The oracle's loop
runs as separately rounded FP32 tensor operations on the GPU: the same bits, in
seconds instead of minutes at these sizes.)"""
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


def process(Wt, k):
    """oracle.ofrr.hessenberg(arith="f32") on the columns Wt[j], in place; the pivots."""
    tol = torch.tensor(O.hessenberg_tol("f32", k), dtype=torch.float32, device="cuda")
    thr = tol * Wt.abs().amax(1)
    piv = []
    for j in range(k):
        r = int(Wt[j].abs().argmax())
        p = Wt[j, r].clone()
        if bool(p.abs() >= thr[j]) and float(p) != 0.0:
            Wt[j] = Wt[j] / p
            for c in range(j + 1, k):
                Wt[c] -= Wt[j] * Wt[c, r].clone()
            piv.append(r)
        else:
            Wt[j] = 0
            piv.append(-1)
    return piv


def test_reference_equals_the_oracle():
    g = torch.Generator(device="cuda").manual_seed(1)
    Wt = torch.randn(9, 5000, generator=g, device="cuda")
    _, pivo, _, Qo = O.hessenberg(Wt.t().cpu().numpy(), arith="f32")
    piv = process(Wt, 9)
    assert piv == list(pivo) and torch.equal(Wt.t().cpu(), torch.from_numpy(Qo))


@pytest.mark.parametrize("n,k", [(9000001, 16), (9000001, 17), (8900000, 37)])
def test_tall_blocks_bitexact(rr, n, k):
    g = torch.Generator(device="cuda").manual_seed(k)
    Wt = torch.randn(k, n, generator=g, device="cuda")
    Wd = Wt.clone().t()
    Q, piv, err = rr.rr_hessenberg(Wd, qtype=torch.float32)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert piv.tolist() == process(Wt, k)
    assert torch.equal(Q, Wt.t()) and torch.equal(Wd, Wt.t())
