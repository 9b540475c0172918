"""The stated error bounds of the FP64-accurate products, on the block that comes
nearest to them: every entry has the digits (65, -64, -64, ..., -64) in base 128,
so nothing is left as a remainder and every dropped pair of digits is as large as
it can be, with one sign.  Exact rational values."""
from fractions import Fraction

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


def entry(digits):
    """65 2^-7 - 64 (2^-14 + ... + 2^(-7 digits)), in (1/2, 1): exact in FP64 for 7 digits."""
    v = Fraction(65, 128) - sum(Fraction(64, 128 ** p) for p in range(2, digits + 1))
    assert Fraction(float(v)) == v
    return v


def block(rows, cols, v):
    return torch.full((cols, rows), float(v), dtype=torch.float64, device="cuda").t()


@pytest.mark.parametrize("K", [64, 448, 1024, 10000])
def test_constant_digits(rr, K):
    v = entry(7)
    exact = K * v * v
    # K 2^-45 max max, and one rounding of the sum per 448 terms and range of K
    bound = Fraction(K, 2 ** 45) * v * v + exact * Fraction(K // 448 + 64, 2 ** 53)
    outs = [rr.rr_gram(block(K, 3, v), block(K, 2, v)),
            rr.rr_gemm_f64_emulated(0, block(8, K, v), block(K, 2, v)),
            rr.rr_gemm_f64_emulated(1, block(K, 8, v), block(K, 2, v))]
    if K <= 512:
        outs.append(rr.rr_lift(block(5, K, v), block(K, 2, v)))
    for C in outs:
        for x in C.flatten().tolist():
            assert abs(Fraction(x) - exact) <= bound, float(abs(Fraction(x) - exact) / bound)
    # 9 digits: 2^-59
    b9 = Fraction(K, 2 ** 59) * v * v + exact * Fraction(K // 352 + 64, 2 ** 53)
    for x in rr.rr_gemm_f64_emulated(0, block(8, K, v), block(K, 2, v), slices=10).flatten().tolist():
        assert abs(Fraction(x) - exact) <= b9
