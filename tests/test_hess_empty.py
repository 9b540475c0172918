"""Algorithm 8 on a block without rows: no crash in the host code that lays out
the launch (it divides by the rows of a CTA), every column skipped."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALL = """
import ctypes, sys
sys.path.insert(0, {root!r})
from paper_2505_00281_gb300 import _lib, build
build.build()
L, RR, p = _lib.lib(), _lib.RR, ctypes.c_void_p(0x1000)
for arith, q in ((RR.F32, RR.F32), (RR.F32, RR.BF16), (RR.F64, RR.F64)):
    print(L.rr_hessenberg(arith, 0, 4, p, 1, q, p, 1, p, ctypes.c_double(0.0), p, 1 << 20, None))
print(L.rr_hessenberg_blocked(0, 4, p, 1, RR.F32, p, 1, p, ctypes.c_double(0.0), 8, p, 1 << 20, None))
print(RR.ERR_CUDA)
"""


@pytest.mark.skipif(torch.cuda.is_available(), reason="fake pointers: must not reach a device")
def test_no_rows_returns_on_the_host():
    # without a GPU the first device call is refused: the calls come back with RR_ERR_CUDA
    r = subprocess.run([sys.executable, "-c", CALL.format(root=ROOT)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    out = [int(x) for x in r.stdout.split()]
    assert out[:-1] == [out[-1]] * 4


@pytest.mark.gpu
@pytest.mark.parametrize("arith,qtype", [("F32", "BF16"), ("F32", "F32"), ("F64", "F64")])
def test_no_rows_skips_every_column(arith, qtype):
    import ctypes

    from paper_2505_00281_gb300 import _lib, build

    build.build()
    L, RR = _lib.lib(), _lib.RR
    buf = torch.zeros(64, dtype=torch.float64, device="cuda")
    piv = torch.zeros(4, dtype=torch.int32, device="cuda")
    ws = torch.ones(1 << 20, dtype=torch.uint8, device="cuda")
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert L.rr_hessenberg(getattr(RR, arith), 0, 4, ptr(buf), 1, getattr(RR, qtype), ptr(buf), 1, ptr(piv),
                           ctypes.c_double(0.0), ptr(ws), ws.numel(), None) == 0
    torch.cuda.synchronize()
    assert piv.tolist() == [-1] * 4 and ws[:4].tolist() == [0] * 4
    if arith == "F32":
        piv.zero_()
        torch.cuda.synchronize()
        assert L.rr_hessenberg_blocked(0, 4, ptr(buf), 1, getattr(RR, qtype), ptr(buf), 1, ptr(piv),
                                       ctypes.c_double(0.0), 8, ptr(ws), ws.numel(), None) == 0
        torch.cuda.synchronize()
        assert piv.tolist() == [-1] * 4
