"""The work whose speed is measured: single steps of the method and whole SVD solves.

A case is a dict of plain values: ``kind`` names the step and the other entries
are its sizes and types.  ``listed()`` gives the standard cases, ``draw(rng)``
one more of the same ranges, ``prepare`` a program's inputs on the GPU, ``run``
one pass through the package's public entry points, ``work`` the bytes and
operations that a pass cannot do without, ``exact`` its outputs in 64-bit
arithmetic where the outputs have such a value.

The kinds and what they stand for:

* ``svd``      rr_svd, the whole mixed-precision solve (BF16 basis, refinement)
               of a dense operator with a known SVD.
* ``lowp``     rr_gemm_lowp, one BF16 product W = A V of the block filter.
* ``f64prod``  rr_gemm_f64_emulated, the FP64-accurate products A X (trans 0)
               and A^T Y (trans 1) behind the residuals.
* ``hess``     rr_hessenberg, the basis step after every product (FP32
               arithmetic; stored BF16, or FP32 for a sweep's last block).
* ``gram``     rr_gram, the projection products of the FP64 Ritz vectors and
               the lower-precision correction blocks.
* ``lift``     rr_lift, the Ritz lift X = [S1 S2] Y.
* ``chebrows`` rr_chebyshev_step_rows, one step of the plain Chebyshev filter
               on the 5-point grid operator (row-major blocks).
* ``chebcols`` rr_chebyshev_step, one step of the refinement's correction
               recurrence on the same operator (column-major, driven by R).
* ``psvd``, ``peig``  rr_pencil_svd and rr_pencil_eig, the small projected problems.
"""
import math

import torch

import paper_2505_00281_gb300 as rr

DEV = "cuda"
TYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest solve a user runs: launches and host steps count
        {"name": "svd 1024x256 b32", "kind": "svd", "m": 1024, "n": 256, "b": 32},
        # the headline solve: top 64 triplets of a 16384 x 4096 operator
        {"name": "svd 16384x4096 b128", "kind": "svd", "m": 16384, "n": 4096, "b": 128},
        # one filter product of that solve
        {"name": "lowp 16384x4096x128", "kind": "lowp", "M": 16384, "N": 128, "K": 4096},
        # its FP64-accurate residual product
        {"name": "f64prod 16384x4096x128", "kind": "f64prod", "trans": 0, "m": 16384, "n": 4096, "N": 128},
        # the transposed product of a mid-sized problem of the batched workload (ragged: no multiple of a tile)
        {"name": "f64prod T 2520x632x32", "kind": "f64prod", "trans": 1, "m": 2520, "n": 632, "N": 32},
        # the basis step of the headline solve's tall side
        {"name": "hess 16384x128", "kind": "hess", "n": 16384, "k": 128, "q": "bf16"},
        # the basis step of the sparse workload (1024 x 1024 grid, block 160)
        {"name": "hess 1048576x160", "kind": "hess", "n": 1048576, "k": 160, "q": "bf16"},
        # the sparse workload's coupling block X^T D of its 2b = 320 pencil
        {"name": "gram 1048576 160x160", "kind": "gram", "n": 1048576, "p": 160, "q": 160, "x": "f64", "y": "bf16"},
        # the lift of a mid-sized grid (odd number of rows) from Ritz vectors and BF16 corrections
        {"name": "lift 360001 96+96", "kind": "lift", "n": 360001, "p1": 96, "p2": 96, "b": 96, "t1": "f64", "t2": "bf16"},
        # the sparse workload's plain filter step
        {"name": "chebrows 1024^2 b160", "kind": "chebrows", "grid": 1024, "b": 160, "t": "bf16"},
        # its correction step on a mid-sized grid, an odd number of columns
        {"name": "chebcols 509^2 b95", "kind": "chebcols", "grid": 509, "b": 95, "t": "bf16", "out": "f32"},
        # the headline solve's refinement pencil (2b = 256)
        {"name": "psvd 256", "kind": "psvd", "b": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["svd", "lowp", "f64prod", "f64prod", "hess", "hess", "gram", "gram", "lift", "lift",
                       "chebrows", "chebcols", "psvd", "peig"])
    if kind == "svd":
        b = rng.choice([16, 24, 32, 48, 64, 96, 128])
        m = _log(rng, 16 * b, 12000)
        return {"kind": kind, "m": m, "n": min(m, max(4 * b, m // rng.choice([2, 3, 4]))), "b": b}
    if kind == "lowp":
        return {"kind": kind, "M": _log(rng, 256, 16384), "N": rng.randint(16, 128), "K": 8 * _log(rng, 32, 512)}
    if kind == "f64prod":
        return {"kind": kind, "trans": rng.randint(0, 1), "m": 8 * _log(rng, 32, 1600), "n": 8 * _log(rng, 16, 400),
                "N": rng.randint(16, 128)}
    if kind == "hess":
        k = rng.randint(16, 160)
        return {"kind": kind, "n": _log(rng, 1024, 900000), "k": k, "q": rng.choice(["bf16", "bf16", "f32"])}
    if kind == "gram":
        x, y = rng.choice([("f64", "f64"), ("f64", "bf16"), ("f64", "f32"), ("bf16", "bf16"), ("bf16", "f64")])
        return {"kind": kind, "n": _log(rng, 256, 125000) * rng.choice([8, 8, 4]), "p": rng.randint(16, 160),
                "q": rng.randint(16, 160), "x": x, "y": y}
    if kind == "lift":
        two = rng.choice([0, 1, 1])
        b = 8 * rng.randint(2, 20)
        return {"kind": kind, "n": _log(rng, 1024, 350000), "p1": b, "p2": b * two, "b": b,
                "t1": rng.choice(["f64", "f64", "bf16"]), "t2": rng.choice(["bf16", "f32", "f64"])}
    if kind == "chebrows":
        return {"kind": kind, "grid": _log(rng, 48, 900), "b": rng.randint(8, 160), "t": rng.choice(["bf16", "bf16", "f32"])}
    if kind == "chebcols":
        t = rng.choice(["bf16", "bf16", "f32"])
        return {"kind": kind, "grid": _log(rng, 48, 700), "b": rng.randint(8, 160), "t": t, "out": "f32"}
    return {"kind": kind, "b": rng.randint(24, 256 if kind == "psvd" else 320)}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, rows, cols, dtype=torch.float64):
    """Column-major N(0, 1) block."""
    return torch.randn(cols, rows, generator=g, device=DEV, dtype=dtype).t()


class _Orthogonal:
    """A dense random orthogonal matrix applied in O(n log n): random signs and
    Hartley transforms, D1 H D2 H D3."""

    def __init__(self, n, g):
        self.d = torch.sign(torch.rand(3, n, generator=g, device=DEV, dtype=torch.float64) - 0.5)
        self.n = n

    def times(self, x):
        """Q x for x with one row per transform (applied along the last dimension)."""
        for i in (2, 1):
            f = torch.fft.fft(x * self.d[i])
            x = (f.real - f.imag) / math.sqrt(self.n)
        return x * self.d[0]


def _svd_parts(case, seed):
    """sigma_i = exp(-i 64 / (30 b)) (the headline decay exp(-i / 60) at b = 128) and the two factors."""
    g = _gen(seed)
    n = case["n"]
    s = torch.exp(-torch.arange(1, n + 1, dtype=torch.float64, device=DEV) * 64.0 / (30.0 * case["b"]))
    return s, _Orthogonal(case["m"], g), _Orthogonal(n, g), g


def _svd_operator(case, seed):
    m, n = case["m"], case["n"]
    s, qu, qv, g = _svd_parts(case, seed)
    rows = qv.times(torch.diag(s))                      # row i: s_i v_i^T
    at = torch.empty(n, m, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 25) // m)
    for j in range(0, n, step):                         # A = U diag(s) V^T by columns: A(:, j) = Qu [diag(s) V^T](:, j)
        e = torch.zeros(min(step, n - j), m, dtype=torch.float64, device=DEV)
        e[:, :n] = rows[:, j:j + step].t()
        at[j:j + step] = qu.times(e)
    return at.t(), torch.rand(case["b"], n, generator=g, device=DEV, dtype=torch.float64).t()


def _grid(case, seed):
    """CSR of -Laplacian + diag(v) on a grid x grid Dirichlet square, v ~ U(0, 10), FP32 values."""
    N = case["grid"]
    n = N * N
    g = _gen(seed)
    diag = 4.0 + 10.0 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    p = torch.arange(n, device=DEV)
    x, y = p % N, p // N
    cols = torch.stack([p - N, p - 1, p, p + 1, p + N], 1)
    one = torch.full((n,), -1.0, dtype=torch.float64, device=DEV)
    vals = torch.stack([one, one, diag, one, one], 1)
    ok = torch.stack([y > 0, x > 0, x >= 0, x < N - 1, y < N - 1], 1)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(ok.sum(1), 0, out=ptr[1:])
    return ptr.to(torch.int32), cols[ok].to(torch.int32), vals[ok].to(torch.float32), diag.float(), g


def _pencil(case, seed):
    """Well-separated values and the factors R of the Grams G = R^T R of two
    non-orthogonal bases (unit columns up to a condition of about 1e3)."""
    b = case["b"]
    g = _gen(seed)
    i = torch.arange(1, b + 1, dtype=torch.float64, device=DEV)
    lam = torch.exp(-i / 60.0) if case["kind"] == "psvd" else 0.1 + 8.0 * i / b
    q = [torch.linalg.qr(torch.randn(b, b, generator=g, device=DEV, dtype=torch.float64))[0] for _ in range(2)]
    f = [torch.eye(b, dtype=torch.float64, device=DEV)
         + 0.6 / math.sqrt(b) * torch.randn(b, b, generator=g, device=DEV, dtype=torch.float64) for _ in range(2)]
    return lam, q, f


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed)
    if kind == "svd":
        A, V0 = _svd_operator(case, seed)
        b = case["b"]
        params = rr.api.make_params(b // 2, b, 4, 30, 1e-10, basis="bf16", v0=V0, refine=True, phase1_sweeps=1)
        return {"kind": kind, "op": rr.api.dense_operator(A), "params": params}
    if kind == "lowp":
        M, N, K = case["M"], case["N"], case["K"]
        A = torch.randn(M, K, generator=g, device=DEV).bfloat16()
        B = torch.randn(N, K, generator=g, device=DEV).bfloat16()
        return {"kind": kind, "size": (M, N, K), "A": A, "B": B.t()}
    if kind == "f64prod":
        m, n = case["m"], case["n"]
        X = _randn(g, n if case["trans"] == 0 else m, case["N"])
        return {"kind": kind, "trans": case["trans"], "A": _randn(g, m, n) / math.sqrt(n), "X": X / X.norm(dim=0)}
    if kind == "hess":
        return {"kind": kind, "W": _randn(g, case["n"], case["k"], torch.float32), "q": TYPES[case["q"]]}
    if kind == "gram":
        X, Y = _randn(g, case["n"], case["p"]), _randn(g, case["n"], case["q"])
        X = (X / X.norm(dim=0)).to(TYPES[case["x"]])
        Y = (Y / Y.abs().amax(dim=0)).to(TYPES[case["y"]])
        return {"kind": kind, "X": X, "Y": Y}
    if kind == "lift":
        S1 = _randn(g, case["n"], case["p1"])
        S1 = (S1 / S1.norm(dim=0)).to(TYPES[case["t1"]])
        S2 = None
        if case["p2"]:
            S2 = _randn(g, case["n"], case["p2"])
            S2 = (S2 / S2.abs().amax(dim=0)).to(TYPES[case["t2"]])
        return {"kind": kind, "S1": S1, "S2": S2, "Y": _randn(g, case["p1"] + case["p2"], case["b"]) / 8.0}
    if kind == "chebrows":
        rp, ci, va, _, g = _grid(case, seed)
        n, b = case["grid"] ** 2, case["b"]
        ldr = -(-b // 8) * 8
        Y = [torch.randn(n, ldr, generator=g, device=DEV).to(TYPES[case["t"]]) for _ in range(2)]
        for y in Y:
            y[:, b:] = 0
        return {"kind": kind, "csr": (rp, ci, va), "Y": Y, "b": b}
    if kind == "chebcols":
        rp, ci, va, _, g = _grid(case, seed)
        n, b = case["grid"] ** 2, case["b"]
        Y = [_randn(g, n, b, torch.float32).to(TYPES[case["t"]]) for _ in range(2)]
        R = _randn(g, n, b)
        f = torch.rand(2, b, generator=g, device=DEV, dtype=torch.float64)
        return {"kind": kind, "csr": (rp, ci, va), "Y": Y, "R": R, "beta": 0.5 + f[0], "gamma": f[1], "out": TYPES[case["out"]]}
    lam, q, f = _pencil(case, seed)
    if kind == "psvd":
        B = f[0].t() @ (q[0] * lam) @ q[1].t() @ f[1]
        return {"kind": kind, "B": rr.fortran(B), "Gu": rr.fortran(f[0].t() @ f[0]), "Gv": rr.fortran(f[1].t() @ f[1])}
    H = f[0].t() @ (q[0] * lam) @ q[0].t() @ f[0]
    return {"kind": kind, "H": rr.fortran((H + H.t()) / 2), "G": rr.fortran(f[0].t() @ f[0])}


# ---------------------------------------------------------------- one pass
# the filter's centre, half width and recurrence coefficients at the grid operator's scale
ALPHA, CENTRE, BETA = 0.21, 9.0, 0.87


def _signed(lead, *others):
    """Vectors are defined up to a sign: the largest entry of each column of `lead` made positive."""
    at = lead.abs().argmax(dim=0, keepdim=True)
    s = torch.sign(lead.gather(0, at))
    return [v * s for v in (lead,) + others]


def run(state):
    kind = state["kind"]
    if kind == "svd":
        s, U, V, info = rr.rr_svd(state["op"], state["params"])
        return {"sigma": s, "U": U, "V": V, "converged": info["n_converged"]}
    if kind == "lowp":
        M, N, K = state["size"]
        return rr.api.rr_gemm_lowp(rr.RR.BF16, M, N, K, state["A"], K, state["B"], K)
    if kind == "f64prod":
        return rr.api.rr_gemm_f64_emulated(state["trans"], state["A"], state["X"])
    if kind == "hess":
        W = state["W"].clone()      # the call overwrites the product it is given
        Q, piv, _ = rr.api.rr_hessenberg(W, state["q"])
        return {"Q": Q, "W": W, "piv": piv}
    if kind == "gram":
        return rr.api.rr_gram(state["X"], state["Y"])
    if kind == "lift":
        return rr.api.rr_lift(state["S1"], state["Y"], state["S2"])
    if kind == "chebrows":
        return rr.api.rr_chebyshev_step_rows(*state["csr"], state["Y"][0], state["Y"][1], state["b"], ALPHA, CENTRE, BETA)
    if kind == "chebcols":
        return rr.api.rr_chebyshev_step(*state["csr"], state["Y"][0], state["Y"][1], ALPHA, CENTRE, BETA, state["beta"],
                                        state["R"], state["gamma"], state["out"])
    if kind == "psvd":
        s, Y, Z, _ = rr.api.rr_pencil_svd(state["B"], state["Gu"], state["Gv"])
        Z, Y = _signed(Z, Y)
        return {"s": s, "Y": Y, "Z": Z}
    theta, Y, _ = rr.api.rr_pencil_eig(state["H"], state["G"])
    return {"theta": theta, "Y": _signed(Y)[0]}


def work(case):
    kind = case["kind"]
    if kind == "svd":
        m, n, b = case["m"], case["n"], case["b"]
        # one sweep of 4 products with A and 4 with A^T, twice: the plain one and at least one refinement
        return {"bytes": 8.0 * (m * n + (m + n) * (b // 2) + n * b), "flops": 2.0 * 8 * 2 * m * n * b}
    if kind == "lowp":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2.0 * (M * K + K * N) + 4.0 * M * N, "flops": 2.0 * M * N * K}
    if kind == "f64prod":
        m, n, N = case["m"], case["n"], case["N"]
        return {"bytes": 8.0 * (m * n + (m + n) * N), "flops": 2.0 * m * n * N}
    if kind == "hess":
        n, k = case["n"], case["k"]
        return {"bytes": n * k * (8.0 + SIZE[case["q"]]), "flops": 1.0 * n * k * k}
    if kind == "gram":
        n, p, q = case["n"], case["p"], case["q"]
        return {"bytes": n * (p * SIZE[case["x"]] + q * SIZE[case["y"]]) + 8.0 * p * q, "flops": 2.0 * n * p * q}
    if kind == "lift":
        n, p1, p2, b = case["n"], case["p1"], case["p2"], case["b"]
        return {"bytes": n * (p1 * SIZE[case["t1"]] + p2 * SIZE[case["t2"]] + 8.0 * b), "flops": 2.0 * n * (p1 + p2) * b}
    if kind in ("chebrows", "chebcols"):
        n, b = case["grid"] ** 2, case["b"]
        csr = 5 * n * 8.0 + 4.0 * n
        if kind == "chebrows":
            return {"bytes": csr + 3.0 * n * b * SIZE[case["t"]], "flops": 13.0 * n * b}
        return {"bytes": csr + n * b * (2.0 * SIZE[case["t"]] + 8 + SIZE[case["out"]]), "flops": 15.0 * n * b}
    b = case["b"]
    if kind == "psvd":
        return {"bytes": 8.0 * (5 * b * b + b), "flops": 14.0 * b ** 3}
    return {"bytes": 8.0 * (3 * b * b + b), "flops": 14.0 * b ** 3 / 2}


# ---------------------------------------------------------------- 64-bit values
def _grid_apply(csr, x):
    """A x in FP64 for a column- or row-major block (n x b) of the grid operator."""
    rp, ci, va = csr
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
    a = torch.sparse_coo_tensor(torch.stack([rows, ci.long()]), va.double(), (n, n))
    return torch.cat([torch.sparse.mm(a, x[:, j:j + 16].double().contiguous()) for j in range(0, x.shape[1], 16)], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "svd":
        s, qu, qv, _ = _svd_parts(case, seed)
        k = case["b"] // 2
        e = torch.zeros(k, case["m"], dtype=torch.float64, device=DEV)
        e[:, :k] = torch.eye(k, dtype=torch.float64, device=DEV)
        U = qu.times(e).t()
        V = qv.times(e[:, :case["n"]].contiguous()).t()
        V, U = _signed(V, U)
        return {"sigma": s[:k], "U": U, "V": V, "converged": None}
    st = prepare(case, seed)
    if kind == "lowp":
        return (st["A"].double() @ st["B"].double())
    if kind == "f64prod":
        return (st["A"].t() if case["trans"] else st["A"]) @ st["X"]
    if kind == "hess":
        # row-pivoted elimination in 64 bits; pivots that FP32 rounding decides otherwise are not comparable
        W = st["W"].double()
        for j in range(case["k"]):
            r = W[:, j].abs().argmax()
            c = W[:, j] / W[r, j]
            w = W[r, j + 1:].clone()
            W[:, j] = c
            W[:, j + 1:].addr_(c, w, alpha=-1.0)
        return {"Q": W, "W": W, "piv": None}
    if kind == "gram":
        return st["X"].double().t() @ st["Y"].double()
    if kind == "lift":
        S = st["S1"].double() if st["S2"] is None else torch.cat([st["S1"].double(), st["S2"].double()], 1)
        return S @ st["Y"]
    if kind == "chebrows":
        y, prev = st["Y"]
        return ALPHA * (_grid_apply(st["csr"], y) - CENTRE * y.double()) - BETA * prev.double()
    if kind == "chebcols":
        y, prev = st["Y"]
        return (ALPHA * (_grid_apply(st["csr"], y) - CENTRE * y.double()) - BETA * st["beta"] * prev.double()
                + st["gamma"] * st["R"])
    lam, q, f = _pencil(case, seed)
    if kind == "psvd":
        Y, Z = torch.linalg.solve(f[0], q[0]), torch.linalg.solve(f[1], q[1])
        Z, Y = _signed(Z, Y)
        return {"s": lam, "Y": Y, "Z": Z}
    return {"theta": lam, "Y": _signed(torch.linalg.solve(f[0], q[0]))[0]}
