"""The work that a user of this library has it do, as cases that can be timed.

Twelve listed cases cover the solver's public entry points over the range
that its tests, benchmark and header use: the products with C = A^T A, the
block Gram-Schmidt pass, the basis transforms, the CSR -> CSC set-up, one
training step of the correction network, and whole solves.  ``draw`` gives
more cases of the same ranges.

Inputs are made on the GPU from the seed alone.  Matrices follow the families
of ``paper_1408_5535_gb300.synth`` (random sparse with Poisson rows, weighted
grid gradients); tall blocks hold columns of unit norm, as an orthonormal
basis does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1408_5535_gb300 import learned, native, synth

TOL = 1e-14
DTYPE = {"f64": torch.float64, "f32": torch.float32}
SIZE = {"f64": 8, "f32": 4}


def listed():
    return [
        # Product with C of the mixed-precision stage 1 on the benchmark's matrix: FP32, block 8, unstructured gathers.
        {"name": "spmm_random_f32_b8", "op": "spmm", "matrix": "random", "m": 1000000, "n": 500000, "row": 12.0,
         "dtype": "f32", "b": 8, "schedule": 2},
        # The same product in FP64 on the 512 x 512 grid gradient: structured, one or two entries per row, block 4.
        {"name": "spmm_grid512_f64_b4", "op": "spmm", "matrix": "grid", "grid": 512, "dtype": "f64", "b": 4,
         "schedule": 2},
        # The allocation-free product of a latency-critical loop: one vector, 32 x 32 grid, a few microseconds.
        {"name": "spmm_static_grid32", "op": "spmm_static", "matrix": "grid", "grid": 32, "b": 1},
        # Second Gram-Schmidt pass of a stage-1 iteration in FP64: 20 locked and 35 basis columns against a block of 8.
        {"name": "cgs_f64_500k", "op": "cgs", "dtype": "f64", "n": 500000, "p1": 20, "p2": 35, "q": 8,
         "sub": True, "gout": True, "tout": False},
        # A pass of the FP32 stage on the 512 x 512 grid: subtract, project, and the Gram of a block of 4.
        {"name": "cgs_f32_262k", "op": "cgs", "dtype": "f32", "n": 262144, "p1": 6, "p2": 29, "q": 4,
         "sub": True, "gout": True, "tout": True},
        # Thick restart V <- V Y in FP64 at the benchmark's size: 35 basis columns to 21.
        {"name": "tall_f64_500k", "op": "tall", "dtype": "f64", "n": 500000, "p": 35, "r": 21, "theta": False,
         "norms": False},
        # Residuals R = W S - X theta with their norms in the FP32 stage, odd length.
        {"name": "tall_f32_155k", "op": "tall", "dtype": "f32", "n": 155649, "p": 35, "r": 8, "theta": True,
         "norms": True},
        # The transposed copy that each solve builds first, at the benchmark's size.
        {"name": "csc_random", "op": "csc", "m": 1000000, "n": 500000, "row": 12.0},
        # One training step (forward, backward, Adam) of the correction network: 32 residual images of 32 x 32.
        {"name": "cnn_step_32x32", "op": "cnn", "batch": 32, "nx": 32, "ny": 32},
        # A small whole solve from host arrays with the default options: latency of the iteration decides.
        {"name": "solve_small_host", "op": "solve", "matrix": "random", "m": 2000, "n": 1000, "row": 8.0, "k": 5,
         "target": "smallest", "block": 1, "precision": "fp64", "device": False, "vectors": True},
        # The smallest triplets of an ill-conditioned PDE matrix by the Jacobi-Davidson path, mixed precision.
        {"name": "solve_grid64_smallest", "op": "solve", "matrix": "grid", "grid": 64, "k": 10, "target": "smallest",
         "block": 4, "precision": "mixed", "device": True, "vectors": False},
        # The benchmark's solve: 20 largest triplets of the 1,000,000 x 500,000 matrix, mixed precision, device arrays.
        {"name": "solve_random_largest", "op": "solve", "matrix": "heavy", "m": 1000000, "n": 500000, "row": 12.0,
         "k": 20, "target": "largest", "block": 8, "precision": "mixed", "device": True, "vectors": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["spmm", "spmm", "spmm_static", "cgs", "cgs", "cgs", "tall", "tall", "tall", "csc", "cnn", "solve"])
    dtype = rng.choice(["f64", "f32"])
    if op == "spmm":
        b = rng.choice([1, 2, 4, 8])
        schedule = rng.choice([1, 2])
        if rng.random() < 0.5:
            return {"op": op, "matrix": "grid", "grid": _log(rng, 17, 512), "dtype": dtype, "b": b,
                    "schedule": schedule}
        n = _log(rng, 1000, 400000)
        return {"op": op, "matrix": "random", "m": n + int(n * rng.uniform(0.2, 1.0)), "n": n,
                "row": round(rng.uniform(3.0, 12.0), 2), "dtype": dtype, "b": b, "schedule": schedule}
    if op == "spmm_static":
        return {"op": op, "matrix": "grid", "grid": _log(rng, 16, 120), "b": rng.choice([1, 2, 4, 8])}
    if op == "cgs":
        q = rng.randint(1, 8)
        p1 = rng.choice([0, rng.randint(1, 20)])
        sub, gout, tout = rng.choice([(False, True, False), (True, True, False), (True, False, True),
                                      (True, True, True)])
        return {"op": op, "dtype": dtype, "n": _log(rng, 1000, 500000), "p1": p1, "p2": rng.randint(4, 40), "q": q,
                "sub": sub, "gout": gout, "tout": tout}
    if op == "tall":
        p = rng.randint(8, 43)
        theta = rng.random() < 0.5
        return {"op": op, "dtype": dtype, "n": _log(rng, 1000, 500000), "p": p,
                "r": rng.randint(1, 10) if theta else rng.randint(1, min(p, 21)), "theta": theta, "norms": theta}
    if op == "csc":
        n = _log(rng, 1000, 400000)
        return {"op": op, "m": n + int(n * rng.uniform(0.0, 1.0)), "n": n, "row": round(rng.uniform(2.0, 12.0), 2)}
    if op == "cnn":
        return {"op": op, "batch": rng.randint(1, 32), "nx": rng.randint(16, 64), "ny": rng.randint(16, 64)}
    if rng.random() < 0.5:
        n = _log(rng, 300, 1500)
        return {"op": op, "matrix": "random", "m": 2 * n + rng.randint(0, 99), "n": n,
                "row": round(rng.uniform(7.0, 12.0), 2), "k": rng.randint(1, 5), "target": "smallest",
                "block": rng.choice([1, 2]), "precision": rng.choice(["fp64", "mixed"]),
                "device": rng.random() < 0.5, "vectors": True}
    n = _log(rng, 5000, 200000)
    return {"op": op, "matrix": "heavy", "m": n + int(n * rng.uniform(0.2, 1.0)), "n": n, "row": 12.0,
            "k": rng.randint(5, 20), "target": "largest", "block": rng.choice([4, 8]),
            "precision": rng.choice(["fp64", "mixed"]), "device": True, "vectors": False}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _random_csr(m, n, row, seed, heavy):
    """Poisson(row) entries per row at uniform columns and the diagonal, _nnz(case) entries in all; heavy: log-normal(2)
    values with random signs and 1e-3 [I; 0], else normal values and a diagonal shift of 0.05."""
    g = _gen(seed)
    counts = torch.poisson(torch.full((m,), float(row) / 0.9, device="cuda"), generator=g).long()
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), counts)
    key = torch.unique(rows * n + torch.randint(0, n, (rows.numel(),), device="cuda", generator=g))
    key = key[(key % n) != key // n]                      # the diagonal is added below
    key = key[torch.randperm(key.numel(), device="cuda", generator=g)[: int(m * row)]]
    diag = torch.arange(n, device="cuda") * (n + 1)
    key = torch.sort(torch.cat([key, diag]))[0]
    val = torch.randn(key.numel(), device="cuda", dtype=torch.float64, generator=g)
    if heavy:
        sign = torch.randint(0, 2, (key.numel(),), device="cuda", generator=g).double() * 2 - 1
        val = sign * torch.exp(2.0 * val)
    val[torch.searchsorted(key, diag)] += 1e-3 if heavy else 0.05
    rows = key // n
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return m, n, rp, (key % n).int(), val


def _matrix(case, seed):
    """(m, n, row_ptr int64, col int32, val float64), on the GPU."""
    if case["op"] == "csc" or case["matrix"] in ("random", "heavy"):
        heavy = case.get("matrix") == "heavy" or (case["op"] in ("spmm", "csc"))
        return _random_csr(case["m"], case["n"], case["row"], seed, heavy)
    A = synth.grid_gradient(case["grid"], 1.0, seed)
    return A.m, A.n, *(torch.from_numpy(x).cuda() for x in (A.row_ptr, A.col, A.val))


def _tall(g, n, c, dt):
    """Column-major n x c block (tensor of shape c x n) with columns of about unit norm."""
    return (torch.randn((c, n), device="cuda", dtype=torch.float64, generator=g) / math.sqrt(n)).to(dt)


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case, "h": native.Handle(0)}
    if op in ("spmm", "spmm_static"):
        m, n, rp, ci, va = _matrix(case, seed)
        nnz, dt, b = va.numel(), DTYPE[case.get("dtype", "f64")], case["b"]
        rp = rp.int()
        cp = torch.empty(n + 1, dtype=torch.int32, device="cuda")
        ri = torch.empty(nnz, dtype=torch.int32, device="cuda")
        cv = torch.empty(nnz, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        native.phsvds_csr_to_csc(s["h"], m, n, nnz, rp, ci, va, cp, ri, cv)
        native.phsvds_sync(s["h"])
        X = (torch.rand((n, b), device="cuda", dtype=torch.float64, generator=_gen(seed + 1)) * 2 - 1).to(dt)
        s.update(m=m, n=n, nnz=nnz, b=b, A=(rp, ci, va.to(dt), cp, ri, cv.to(dt)), X=X, Y=torch.empty_like(X),
                 Z=torch.empty((m, b), device="cuda", dtype=dt))
    elif op == "cgs":
        n, p, q, dt = case["n"], case["p1"] + case["p2"], case["q"], DTYPE[case["dtype"]]
        g = _gen(seed)
        P, T = _tall(g, n, p, dt), _tall(g, n, q, dt)
        G = torch.mm(T.double(), P.double().t()).contiguous()          # P^T T, column-major p x q
        out = torch.zeros(p * q + q * q, dtype=torch.float64, device="cuda")
        s.update(n=n, p=p, P=P, T=T, G=G, out=out, Gout=out[: p * q], Tout=out[p * q:])
    elif op == "tall":
        n, p, r, dt = case["n"], case["p"], case["r"], DTYPE[case["dtype"]]
        g = _gen(seed)
        Y = torch.linalg.qr(torch.randn((p, p), device="cuda", dtype=torch.float64, generator=g))[0]
        s.update(n=n, P=_tall(g, n, p, dt), Y=Y.t()[:r].contiguous(), Out=torch.empty((r, n), dtype=dt, device="cuda"),
                 X=_tall(g, n, r, dt) if case["theta"] else None,
                 theta=torch.rand(r, device="cuda", dtype=torch.float64, generator=g) * 3 if case["theta"] else None,
                 norms=torch.zeros(r, dtype=torch.float64, device="cuda") if case["norms"] else None)
    elif op == "csc":
        m, n, rp, ci, va = _matrix(case, seed)
        s.update(m=m, n=n, nnz=va.numel(), A=(rp.int(), ci, va),
                 out=(torch.empty(n + 1, dtype=torch.int32, device="cuda"), torch.empty_like(ci), torch.empty_like(va)))
    elif op == "cnn":
        s.update(_cnn_state(case, seed))
        B, npix = case["batch"], case["nx"] * case["ny"]
        s["y"] = torch.empty((B, case["ny"], case["nx"]), device="cuda")
        s["work"] = torch.empty(native.cnn_work_floats(B, npix), device="cuda")
    else:
        m, n, rp, ci, va = _matrix(case, seed)
        if not case["device"]:
            rp, ci, va = (x.cpu().numpy() for x in (rp, ci, va))
        mixed = native.MIXED if case["precision"] == "mixed" else native.FP64
        if case["matrix"] == "grid":      # ill-conditioned: the Jacobi-Davidson forms of both stages
            o = native.default_opts(block_size=case["block"], precision=mixed, mixed_inner=2, stage2_inner=1,
                                    norm_A=-1.0)
            prec = native.PREC_JACOBI
        else:
            o, prec = native.default_opts(block_size=case["block"], precision=mixed), native.PREC_NONE
        s.update(m=m, n=n, A=(rp, ci, va), opts=o, prec=prec)
    torch.cuda.synchronize()
    return s


def _cnn_state(case, seed):
    """A network and Adam state in the middle of training (step 11), images and unit-RMS targets."""
    g = _gen(seed)
    B, nx, ny = case["batch"], case["nx"], case["ny"]
    w = torch.from_numpy(learned.init_params(seed, last_scale=1.0)).cuda()
    x = torch.randn((B, 4, ny, nx), device="cuda", generator=g)
    x[:, 2:] = (torch.rand((B, 2, 1, 1), device="cuda", generator=g) * 2 - 1)      # constant beta planes
    t = torch.randn((B, ny, nx), device="cuda", generator=g)
    m1 = torch.randn(w.shape, device="cuda", generator=g) * 1e-2
    m2 = (torch.rand(w.shape, device="cuda", generator=g) + 0.5) * 1e-3
    return {"w": w, "params": w.to(torch.bfloat16), "x": x, "t": t, "m1": m1, "m2": m2, "step": 11,
            "grad": torch.zeros_like(w), "loss": torch.zeros(1, dtype=torch.float64, device="cuda")}


# ---------------------------------------------------------------- one pass
def run(s):
    op, h, case = s["op"], s["h"], s["case"]
    if op == "spmm":
        native.phsvds_ata_spmm(h, case["schedule"], s["m"], s["n"], s["nnz"], *s["A"], s["b"], s["X"], s["Y"], s["Z"],
                               fp32=case["dtype"] == "f32")
        return s["Y"]
    if op == "spmm_static":
        native.phsvds_ata_spmm_static(h, s["m"], s["n"], s["nnz"], *s["A"], s["b"], s["X"], s["Y"])
        return s["Y"]
    if op == "cgs":
        n, p1, q = s["n"], case["p1"], case["q"]
        s["out"].zero_()                                   # the call accumulates
        native.phsvds_block_cgs(h, n, s["P"][:p1] if p1 else None, n, p1, s["T"], n, q,
                                Gsub=s["G"] if case["sub"] else None, Gout=s["Gout"] if case["gout"] else None,
                                Tout=s["Tout"] if case["tout"] else None, P2=s["P"][p1:], ld2=n, p2=case["p2"],
                                fp32=case["dtype"] == "f32")
        return s["T"], s["Gout"], s["Tout"]
    if op == "tall":
        n = s["n"]
        if s["norms"] is not None:
            s["norms"].zero_()                             # the call accumulates
        native.phsvds_tall_small(h, n, s["P"], n, case["p"], s["Y"], case["p"], case["r"], s["Out"], n, Xs=s["X"],
                                 ldx=n, theta=s["theta"], norms2=s["norms"], fp32=case["dtype"] == "f32")
        return s["Out"], s["norms"]
    if op == "csc":
        native.phsvds_csr_to_csc(h, s["m"], s["n"], s["nnz"], *s["A"], *s["out"])
        return s["out"]
    if op == "cnn":
        B, nx, ny = case["batch"], case["nx"], case["ny"]
        s["loss"].zero_()
        native.phsvds_cnn_forward(h, B, nx, ny, s["params"], s["x"], s["y"], s["work"])
        native.phsvds_cnn_backward(h, B, nx, ny, s["params"], s["x"], s["y"], s["t"], s["work"], s["grad"], s["loss"])
        native.phsvds_cnn_adam(h, s["w"], s["grad"], s["m1"], s["m2"], s["step"], 1e-3, s["params"])
        s["step"] += 1
        return s["y"], s["loss"], s["w"], s["m1"], s["m2"], s["params"]
    target = native.SMALLEST if case["target"] == "smallest" else native.LARGEST
    # The residuals that come back too are of the size of rounding (1e-15 ||A||), so their digits say nothing.
    sigma, U, V, _, _, _ = native.phsvds_solve(h, s["m"], s["n"], *s["A"], case["k"], target, TOL, s["prec"],
                                               s["opts"], on_device=case["device"], want_vectors=case["vectors"])
    if not case["vectors"]:
        return sigma
    sign = np.sign(V[np.argmax(np.abs(V), axis=0), np.arange(case["k"])])   # a triplet is defined up to its sign
    return sigma, U * sign, V * sign


# ---------------------------------------------------------------- what a pass cannot do without
def _nnz(case):
    if case.get("matrix") == "grid":
        return 4 * case["grid"] ** 2, 2 * case["grid"] * (case["grid"] + 1), case["grid"] ** 2
    return int(case["m"] * case["row"]) + case["n"], case["m"], case["n"]


def work(case):
    op = case["op"]
    w = SIZE.get(case.get("dtype"), 8)
    if op in ("spmm", "spmm_static"):
        nnz, m, n = _nnz(case)
        b = case["b"]
        return {"bytes": nnz * (w + 4) + 4 * (m + 1) + 2 * w * n * b, "flops": 4 * nnz * b}
    if op == "cgs":
        n, p, q = case["n"], case["p1"] + case["p2"], case["q"]
        return {"bytes": w * n * (p + q * (2 if case["sub"] else 1)),
                "flops": 2 * n * p * q * (case["sub"] + case["gout"]) + (n * q * (q + 1) if case["tout"] else 0)}
    if op == "tall":
        n, p, r = case["n"], case["p"], case["r"]
        return {"bytes": w * n * (p + r * (2 if case["theta"] else 1)),
                "flops": 2 * n * p * r + (2 * n * r if case["theta"] else 0) + (2 * n * r if case["norms"] else 0)}
    if op == "csc":
        nnz, m, n = _nnz(case)
        return {"bytes": 24 * nnz + 4 * (m + n + 2), "flops": 0}
    if op == "cnn":
        pix, par = case["batch"] * case["nx"] * case["ny"], native.CNN_NPARAM
        # images, targets and outputs; forward, weight-gradient and input-gradient products
        return {"bytes": 4 * pix * 6 + par * 30, "flops": 2 * pix * (2 * par + par - 576)}
    nnz, m, n = _nnz(case)
    k = case["k"]
    # the matrix once, the triplets once; at least one product with C per triplet and its residual
    return {"bytes": 12 * nnz + 8 * (m + 1) + 8 * k * ((m + n) if case["vectors"] else 1), "flops": 8 * nnz * k}


# ---------------------------------------------------------------- the same in 64 bits, by torch alone
def _spmm64(m, n, rp, ci, va, X):
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), rp[1:] - rp[:-1])
    c = ci.long()
    Z = torch.zeros((m, X.shape[1]), dtype=torch.float64, device="cuda")
    Y = torch.zeros((n, X.shape[1]), dtype=torch.float64, device="cuda")
    for j in range(X.shape[1]):
        Z[:, j].index_add_(0, rows, va * X[c, j])
        Y[:, j].index_add_(0, c, va * Z[rows, j])
    return Y


def exact(case, seed):
    op = case["op"]
    if op in ("spmm", "spmm_static"):
        m, n, rp, ci, va = _matrix(case, seed)
        dt = DTYPE[case.get("dtype", "f64")]
        X = (torch.rand((n, case["b"]), device="cuda", dtype=torch.float64, generator=_gen(seed + 1)) * 2 - 1).to(dt)
        return _spmm64(m, n, rp, ci, va.to(dt).double(), X.double())
    if op == "cgs":
        n, p, q, dt = case["n"], case["p1"] + case["p2"], case["q"], DTYPE[case["dtype"]]
        g = _gen(seed)
        P, T = _tall(g, n, p, dt).double(), _tall(g, n, q, dt).double()
        G = torch.mm(T, P.t())
        if case["sub"]:
            T = T - torch.mm(G, P)
        zero = torch.zeros
        return (T, torch.mm(T, P.t()).reshape(-1) if case["gout"] else zero(p * q, dtype=torch.float64),
                torch.mm(T, T.t()).reshape(-1) if case["tout"] else zero(q * q, dtype=torch.float64))
    if op == "tall":
        n, p, r, dt = case["n"], case["p"], case["r"], DTYPE[case["dtype"]]
        g = _gen(seed)
        Y = torch.linalg.qr(torch.randn((p, p), device="cuda", dtype=torch.float64, generator=g))[0].t()[:r]
        Out = torch.mm(Y, _tall(g, n, p, dt).double())
        if case["theta"]:
            X = _tall(g, n, r, dt).double()
            th = torch.rand(r, device="cuda", dtype=torch.float64, generator=g) * 3
            Out = Out - X * th[:, None]
        return Out, (Out * Out).sum(1) if case["norms"] else None
    if op == "csc":
        m, n, rp, ci, va = _matrix(case, seed)
        rows = torch.repeat_interleave(torch.arange(m, device="cuda"), rp[1:] - rp[:-1])
        order = torch.argsort(ci.long() * m + rows)
        cp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        cp[1:] = torch.cumsum(torch.bincount(ci.long(), minlength=n), 0)
        return cp.int(), rows[order].int(), va[order]
    if op == "cnn":
        return _cnn_exact(case, seed)
    if case["matrix"] == "heavy" or case.get("grid", 0) > 64:
        return None                        # no dense matrix of that size
    m, n, rp, ci, va = _matrix(case, seed)
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), rp[1:] - rp[:-1])
    D = torch.zeros((m, n), dtype=torch.float64, device="cuda")
    D[rows, ci.long()] = va
    if not case["vectors"]:
        return torch.linalg.svdvals(D).flip(0)[: case["k"]]
    U, S, Vt = torch.linalg.svd(D, full_matrices=False)
    k = case["k"]
    U, V = U.flip(1)[:, :k], Vt.flip(0)[:k].t()
    sign = torch.sign(V[V.abs().argmax(0), torch.arange(k, device="cuda")])
    return S.flip(0)[:k], U * sign, V * sign


def _cnn_exact(case, seed):
    s = _cnn_state(case, seed)
    w16 = s["params"].double()
    shapes, W, at = [(16, 4, 3, 3), (16, 16, 3, 3), (1, 16, 3, 3)], [], 0
    for sh in shapes:
        W.append(w16[at: at + math.prod(sh)].reshape(sh).clone().requires_grad_(True))
        at += math.prod(sh)

    def conv(a, w):                        # 3 x 3 correlation with zero padding, as a sum of shifted products
        ny, nx = a.shape[2:]
        a = torch.nn.functional.pad(a, (1, 1, 1, 1))
        return sum(torch.einsum("bcyx,oc->boyx", a[:, :, i: i + ny, j: j + nx], w[:, :, i, j])
                   for i in range(3) for j in range(3))

    y = conv(torch.relu(conv(torch.relu(conv(s["x"].double(), W[0])), W[1])), W[2])[:, 0]
    t = s["t"].double()
    loss = (((y - t) ** 2).sum((1, 2)) / (t ** 2).sum((1, 2))).mean()
    loss.backward()
    g = torch.cat([w.grad.reshape(-1) for w in W])
    m1 = 0.9 * s["m1"].double() + 0.1 * g
    m2 = 0.999 * s["m2"].double() + 0.001 * g * g
    w = s["w"].double() - 1e-3 * (m1 / (1 - 0.9 ** 11)) / (torch.sqrt(m2 / (1 - 0.999 ** 11)) + 1e-8)
    return y.detach(), loss.detach().reshape(1), w, m1, m2, w
