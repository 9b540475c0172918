"""Grams of row counts and lifts of column counts that are no multiple of 8 run
in FP64 arithmetic: the error of an entry is relative to the terms it sums, not
to the largest entries of its columns, infinities follow IEEE rules in a lift,
and subnormals count.

Bound: a sum of K products in FP64 with any order of additions,
    K u64 (|A||B|)_ij  (+ K times the smallest subnormal)."""
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


def dev(a, t="f64"):
    return torch.from_numpy(np.ascontiguousarray(a.T)).to("cuda").to(DT[t]).t()


def host(t):
    return t.detach().double().cpu().numpy()


def check(C, A, B):
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    K = A.shape[1]
    bound = K * 2.0 ** -53 * (np.abs(A).astype(np.longdouble) @ np.abs(B)) + K * np.longdouble(2.0) ** -1074
    err = np.abs(C.astype(np.longdouble) - ref)
    assert np.all(err <= bound), float((err / bound).max())


def apart(rng, n, c, at):
    """Columns whose few largest entries (2^40 times the others) sit in rows `at`."""
    X = rng.standard_normal((n, c))
    X[at] *= 2.0 ** 40
    return X


@pytest.mark.parametrize("n,p,q,xt,yt", [(65, 1, 1, "f64", "f64"), (1001, 17, 130, "f64", "bf16"),
                                         (5003, 128, 65, "bf16", "f64"), (30004, 24, 24, "f64", "f32")])
def test_gram_error_is_relative_to_its_terms(rr, n, p, q, xt, yt):
    rng = np.random.default_rng(n)
    X, Y = apart(rng, n, p, slice(0, 3)), apart(rng, n, q, slice(5, 9))
    Y[0:3] = 0.0
    X[5:9] = 0.0
    X, Y = dev(X, xt), dev(Y, yt)
    check(host(rr.rr_gram(X, Y)), host(X).T, host(Y))


@pytest.mark.parametrize("n,p1,p2,b,t1,t2", [(300, 13, 0, 5, "f64", "f64"), (1000, 33, 32, 17, "f64", "bf16"),
                                             (2049, 100, 101, 48, "bf16", "f64"), (129, 3, 0, 8, "f32", "f64")])
def test_lift_error_is_relative_to_its_terms(rr, n, p1, p2, b, t1, t2):
    rng = np.random.default_rng(n)
    S, Y = rng.standard_normal((n, p1 + p2)), rng.standard_normal((p1 + p2, b))
    S[:, 1] *= 2.0 ** 40        # the largest entry of every row meets a zero
    Y[1] = 0.0
    S1, S2 = dev(S[:, :p1], t1), dev(S[:, p1:], t2) if p2 else None
    A = host(S1) if S2 is None else np.hstack([host(S1), host(S2)])
    check(host(rr.rr_lift(S1, dev(Y), S2)), A, Y)


def test_lift_infinity_and_subnormals(rr):
    rng = np.random.default_rng(4)
    S, Y = rng.standard_normal((200, 9)), np.abs(rng.standard_normal((9, 4))) + 0.5
    S[7, 2], S[11, 3] = np.inf, -np.inf
    X = host(rr.rr_lift(dev(S), dev(Y)))
    assert (X[7] == np.inf).all() and (X[11] == -np.inf).all()
    assert np.isfinite(np.delete(X, (7, 11), 0)).all()
    S = np.full((100, 9), 2.0 ** -1070)
    assert (host(rr.rr_lift(dev(S), dev(np.ones((9, 4))))) == 9 * 2.0 ** -1070).all()


def test_gram_subnormals(rr):
    X, Y = np.full((101, 3), 2.0 ** -1060), np.ones((101, 2))
    assert (host(rr.rr_gram(dev(X), dev(Y))) == 101 * 2.0 ** -1060).all()
