"""FP64-accurate products, lifts and Grams with the operands sliced on chip
(k_emu_mm.cu), at the edges of its tiles, K stages and storage types, against
the product in extended precision.

Bound per entry: an operand keeps 2^-49 of its row's or column's largest entry
(the truncation both sides contribute, summed over K) and the dropped digit
pairs stay below 2^-47 K of both, plus FP64 roundings of the sum:
    2^-46 K max|a_i| max|b_j| + 4 u64 K (|A||B|)_ij."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


def dev(a, t="f64", ld=None):
    """Column-major device block, optionally with a longer leading dimension."""
    rows, cols = a.shape
    ld = ld or rows
    buf = torch.zeros(cols, ld, dtype=DT[t], device="cuda")
    buf[:, :rows] = torch.from_numpy(np.ascontiguousarray(a.T)).to("cuda").to(DT[t])
    return buf.t()[:rows]


def host(t):
    return t.detach().double().cpu().numpy()


def check(C, A, B):
    """C against A B (A m x K, B K x n) in extended precision."""
    K = A.shape[1]
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    bound = (2.0 ** -46 * K * np.outer(np.abs(A).max(1), np.abs(B).max(0))
             + 4 * 2.0 ** -53 * K * (np.abs(A) @ np.abs(B)))
    err = np.abs(C.astype(np.longdouble) - ref)
    assert np.all(err <= bound), float((err / np.maximum(bound, 1e-300)).max())


def block(rng, n, c, scale):
    return rng.standard_normal((n, c)) * np.exp2(rng.integers(-scale, scale + 1, c))[None, :]


@pytest.mark.parametrize("n,p,q,xt,yt,pad", [
    (64, 1, 1, "f64", "f64", 0), (65, 17, 130, "f64", "bf16", 0), (449, 160, 160, "f64", "f64", 1),
    (447, 129, 64, "bf16", "f64", 3), (1000, 192, 33, "f32", "bf16", 0), (5003, 128, 65, "f64", "f32", 2),
    (70001, 20, 16, "bf16", "bf16", 1), (3000, 300, 200, "f64", "f64", 0)])
def test_gram_edges(rr, n, p, q, xt, yt, pad):
    rng = np.random.default_rng(n + p)
    X, Y = dev(block(rng, n, p, 20), xt, n + pad), dev(block(rng, n, q, 20), yt, n + pad)
    G0 = np.asfortranarray(rng.standard_normal((p, q)) * 2.0 ** -20)
    G = rr.rr_gram(X, Y)
    check(host(G), host(X).T, host(Y))
    Gd = dev(G0)
    rr.rr_gram(X, Y, G=Gd, accumulate=True)
    assert np.abs(host(Gd) - (host(G) + G0)).max() <= 2.0 ** -52 * np.abs(host(Gd)).max()


@pytest.mark.parametrize("n,p1,p2,b,t1,t2", [
    (1, 1, 0, 1, "f64", "f64"), (129, 5, 0, 3, "f64", "f64"), (300, 33, 31, 17, "f64", "bf16"),
    (4099, 160, 160, 160, "f64", "bf16"), (1000, 256, 256, 250, "f32", "f64"), (257, 449, 1, 48, "bf16", "f32")])
def test_lift_edges(rr, n, p1, p2, b, t1, t2):
    rng = np.random.default_rng(n + b)
    S1 = dev(rng.standard_normal((n, p1)) * np.exp2(rng.integers(-15, 16, (n, 1))), t1)
    S2 = dev(rng.standard_normal((n, p2)), t2) if p2 else None
    Y = dev(block(rng, p1 + p2, b, 20))
    X = host(rr.rr_lift(S1, Y, S2))
    Yh = host(Y)
    if S2 is None:
        return check(X, host(S1), Yh)
    # the two blocks are scaled on their own: the bounds add up
    K = p1 + p2
    S = np.hstack([host(S1), host(S2)])
    ref = S.astype(np.longdouble) @ Yh.astype(np.longdouble)
    bound = 4 * 2.0 ** -53 * K * (np.abs(S) @ np.abs(Yh))
    for blk, y in ((host(S1), Yh[:p1]), (host(S2), Yh[p1:])):
        bound += 2.0 ** -46 * K * np.outer(np.abs(blk).max(1), np.abs(y).max(0))
    assert np.all(np.abs(X - ref) <= bound)


@pytest.mark.parametrize("trans,m,n,N", [(0, 8, 8, 1), (1, 8, 8, 1), (0, 136, 456, 65), (1, 2520, 632, 32),
                                         (0, 136, 7200, 130), (1, 40000, 64, 16)])
@pytest.mark.parametrize("slices", [8, 10])
def test_product_edges(rr, trans, m, n, N, slices):
    rng = np.random.default_rng(m + N)
    A = dev(rng.standard_normal((m, n)) * np.exp2(rng.integers(-9, 10, (m, n))))
    B = dev(block(rng, m if trans else n, N, 20))
    C = host(rr.rr_gemm_f64_emulated(trans, A, B, slices=slices))
    check(C, host(A).T if trans else host(A), host(B))


def test_extreme_scales_zero_columns_and_nonfinite(rr):
    """Columns near the lowest and highest exponents of their type, zero columns, FP32 and BF16
    subnormals; an infinity makes its own row (or column) NaN and no other."""
    rng = np.random.default_rng(5)
    n = 700
    X = rng.standard_normal((n, 8))
    X[rng.random((n, 8)) < 0.3] = 0.0
    X *= 2.0 ** np.array([-1000, -960, -500, 0, 300, 900, 0, 0])
    X[:, 6] = 0.0
    Y = rng.standard_normal((n, 5)) * 2.0 ** np.array([0, 20, -30, 90, 0])
    Y[:, 4] = 0.0
    check(host(rr.rr_gram(dev(X), dev(Y))), X.T, Y)
    for t in ("f32", "bf16"):
        Z = dev(rng.standard_normal((n, 6)) * 2.0 ** np.array([-130, -126, -70, -50, 0, 100]), t)
        check(host(rr.rr_gram(Z, dev(Y))), host(Z).T, Y)
        check(host(rr.rr_lift(Z, dev(Y[:6]))), host(Z), Y[:6])
    X[13, 3] = np.inf
    G = host(rr.rr_gram(dev(X), dev(Y)))
    assert np.isnan(G[3]).all() and np.isfinite(np.delete(G, 3, 0)).all()
