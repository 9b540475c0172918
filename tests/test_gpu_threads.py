"""Two host threads, each with its own stream and workspace, run the same kernel
on blocks of very different sizes side by side: neither's shared-memory limit
may disturb the other's launches."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import paper_2505_00281_gb300 as pkg
    from paper_2505_00281_gb300 import build

    build.build()
    return pkg


def run_threads(jobs):
    """Each job(stream) in a thread of its own; re-raises what a thread raised."""
    errors = []

    def body(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                job(torch.cuda.current_stream())
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


@pytest.mark.parametrize("sizes", [((16384, 128), (5000, 8)), ((4096, 200), (1000, 8))])
def test_hessenberg_in_two_threads(rr, sizes):
    out, ref = [None, None], [None, None]

    def job(i):
        n, k = sizes[i]
        W0 = torch.randn(k, n, generator=torch.Generator(device="cuda").manual_seed(i), device="cuda").t()
        ref[i] = W0.t().clone().t()
        rr.rr_hessenberg(ref[i], qtype=torch.float32)
        torch.cuda.synchronize()

        def go(stream):
            for _ in range(150):
                W = W0.t().clone().t()
                Q, _, err = rr.rr_hessenberg(W, qtype=torch.float32, stream=stream)
            stream.synchronize()
            assert int(err.item()) == 0
            out[i] = Q
        return go

    run_threads([job(0), job(1)])
    for i in (0, 1):
        assert torch.equal(out[i], ref[i])


def test_pencils_in_two_threads(rr):
    out, ref = [None, None], [None, None]

    def job(i, b):
        g = torch.Generator(device="cuda").manual_seed(b)
        eye = rr.fortran(torch.eye(b, dtype=torch.float64, device="cuda"))
        B = rr.fortran(torch.randn(b, b, generator=g, device="cuda", dtype=torch.float64))
        ref[i] = rr.rr_pencil_svd(B, eye, eye)[0]
        torch.cuda.synchronize()

        def go(stream):
            for _ in range(40):
                out[i] = rr.rr_pencil_svd(B, eye, eye, stream=stream)[0]
        return go

    run_threads([job(0, 200), job(1, 40)])
    for i in (0, 1):
        assert torch.equal(out[i], ref[i])
