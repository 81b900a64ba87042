"""The work that programs have this library do, as measurable cases.

The library multiplies sparse graphs with dense blocks (SpMM), works on tall-and-skinny blocks
(Gram, update, combine, re-orthogonalisation), solves for eigenpairs and singular triplets with
these, and trains and applies a small network that proposes start blocks.  Each kind of case goes
through the public functions of paper_1602_01421_gb300:

  spmm     Y = A X of a resident graph, of its transpose, or of a graph streamed from host memory
  block    block_gram, block_update, block_update_gram or block_combine
  expand   one Krylov expansion: W = A V_last, then W orthonormalised against V (spmm, block_orth)
  eigs     a whole eigenvalue solve
  svds     a whole singular value solve of a directed graph
  mlp      the start-block network: forward, or loss and gradient

Graphs are R-MAT (0.57/0.19/0.19/0.05, 16 draws per vertex, relabelled at random), the stand-in
for web and social graphs that the tests and the benchmark use.  The number of vertices need not
be a power of two here: the 2^k ids that R-MAT draws are scaled down to n.
"""
import math

import numpy as np
import torch

import paper_1602_01421_gb300 as fe

DT = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # SpMM of a graph of a thousand vertices: the latency of one call (launches, marshalling)
        {"name": "spmm_tiny_f64_b1", "kind": "spmm", "op": "n", "n": 1000, "b": 1, "dt": "f64"},
        # the first phase of a mixed-precision solve of an ordinary graph
        {"name": "spmm_f32_b4", "kind": "spmm", "op": "n", "n": 1 << 20, "b": 4, "dt": "f32"},
        # the FP64 solve's operator on the benchmark's graph size (4.2 million vertices)
        {"name": "spmm_f64_b4_large", "kind": "spmm", "op": "n", "n": 1 << 22, "b": 4, "dt": "f64"},
        # a graph larger than the device memory granted to it: its panels stream from host memory
        {"name": "spmm_streamed_f32_b4", "kind": "spmm", "op": "semi", "n": 1 << 20, "b": 4, "dt": "f32"},
        # MvTransMv against a full subspace of 9 blocks, an odd number of rows
        {"name": "gram_f64", "kind": "block", "op": "gram", "n": 3000017, "nv": 9, "b": 4, "nout": 1, "dt": "f64"},
        # the restart product: 8 blocks into 5
        {"name": "combine_f64", "kind": "block", "op": "combine", "n": 1 << 20, "nv": 8, "b": 4, "nout": 5, "dt": "f64"},
        # the second Gram-Schmidt pass of the FP32 phase at the benchmark's size
        {"name": "update_gram_f32", "kind": "block", "op": "update_gram", "n": 1 << 22, "nv": 7, "b": 4, "nout": 1, "dt": "f32"},
        # one expansion step as a program with its own Krylov loop makes it
        {"name": "expand_f64", "kind": "expand", "n": 1 << 20, "nv": 7, "b": 4, "dt": "f64"},
        # the small configuration of the benchmark: 8 eigenpairs in FP64, subspace 32
        {"name": "eigs_f64_small", "kind": "eigs", "n": 1 << 14, "nev": 8, "b": 4, "nb": 8, "mode": "fp64"},
        # many eigenpairs: 32 with the paper's setting of as many blocks (subspace 128), mixed
        {"name": "eigs_mixed_many", "kind": "eigs", "n": 200003, "nev": 32, "b": 4, "nb": 32, "mode": "mixed"},
        # 8 singular triplets of a directed graph, the paper's block 2 and 16 blocks
        {"name": "svds_f64", "kind": "svds", "n": 1 << 18, "nev": 8, "b": 2, "nb": 16, "mode": "fp64"},
        # one gradient of the start-block network on one graph's vertices
        {"name": "mlp_grad", "kind": "mlp", "op": "span", "n": 262141, "h": 64, "b": 4, "t": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmm", "spmm", "spmm", "block", "block", "block", "expand", "eigs", "svds", "mlp"])
    dt = rng.choice(["f32", "f64"])
    if kind == "spmm":
        b = rng.choice([1, 2, 4, 8, 16])
        op = rng.choice(["n", "n", "n", "t", "semi"])
        hi = (1 << 22) if b <= 4 else (1 << 22) * 4 // b
        return {"kind": kind, "op": op, "n": _log(rng, 700 if op != "semi" else 50000, hi if op == "n" else hi // 4),
                "b": b, "dt": dt}
    if kind == "block":
        b = rng.choice([1, 2, 4, 8])
        nv = rng.randint(1, min(16, 64 // b))
        op = rng.choice(["gram", "update", "update_gram", "combine"])
        nout = rng.randint(1, max(1, min(nv, 32 // b))) if op == "combine" else 1
        return {"kind": kind, "op": op, "n": _log(rng, 900, min(1 << 22, (36 << 22) // (b * (nv + nout)))),
                "nv": nv, "b": b, "nout": nout, "dt": dt}
    if kind == "expand":
        b = rng.choice([1, 2, 4, 8])
        return {"kind": kind, "n": _log(rng, 900, 1 << 20), "nv": rng.randint(1, 32 // b), "b": b, "dt": dt}
    if kind == "eigs":
        nev, b, nb = rng.choice([(8, 4, 8), (4, 4, 6), (8, 4, 12), (16, 4, 16), (32, 4, 32), (8, 8, 8), (6, 2, 16)])
        return {"kind": kind, "n": _log(rng, 2000, 50000), "nev": nev, "b": b, "nb": nb,
                "mode": rng.choice(["fp64", "mixed"])}
    if kind == "svds":
        nev = rng.choice([4, 8])
        return {"kind": kind, "n": _log(rng, 2000, 1 << 18), "nev": nev, "b": 2, "nb": 2 * nev,
                "mode": rng.choice(["fp64", "mixed"])}
    op = rng.choice(["forward", "column", "span"])
    b, t = rng.choice([(4, 4), (4, 8), (8, 8)])
    h = 64 if op == "span" else rng.choice([32, 64])
    return {"kind": kind, "op": op, "n": _log(rng, 900, 1 << 18), "h": h, "b": b, "t": t}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)


def _rmat(n, g, directed):
    """(rowptr int64, colidx int64) on the GPU: sorted rows, no loops, no duplicates."""
    bits = max(1, (n - 1).bit_length())
    e = 16 * n
    u = torch.zeros(e, dtype=torch.int64, device="cuda")
    v = torch.zeros(e, dtype=torch.int64, device="cuda")
    for _ in range(bits):
        r = torch.rand(e, generator=g, device="cuda")
        u = 2 * u + (r >= 0.76)
        v = 2 * v + ((r >= 0.57) & (r < 0.76) | (r >= 0.95))
    label = torch.randperm(n, generator=g, device="cuda")
    u, v = label[(u * n) >> bits], label[(v * n) >> bits]
    keep = u != v
    u, v = u[keep], v[keep]
    key = u * n + v if directed else torch.cat([u * n + v, v * n + u])
    del u, v, keep
    key = torch.unique(key)
    rows = key // n
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return ptr, key - rows * n


def _graph(case, seed):
    directed = case["kind"] == "svds" or case.get("op") == "t"
    return _rmat(case["n"], _gen(seed), directed)


def _handle(case, ptr, col):
    kw = {}
    if case["kind"] == "svds" or case.get("op") == "t":
        kw["transpose"] = True
    if case.get("op") == "semi":
        kw["device_mem_cap_bytes"] = int(col.numel())  # a quarter of the plain column indices
    return fe.Csr(ptr.cpu().numpy(), col.to(torch.int32).cpu().numpy(), **kw)


def _normal(seed, *shape, dt=torch.float64, salt=0):
    return torch.randn(*shape, generator=_gen(seed * 31 + 7 + salt), device="cuda", dtype=dt)


def _basis(seed, n, k, salt=0):
    """n x k with orthonormal columns (Cholesky QR, twice), FP64."""
    q = _normal(seed, n, k, salt=salt)
    for _ in range(2):
        q = torch.linalg.solve_triangular(torch.linalg.cholesky(q.T @ q).mT, q, upper=True, left=False)
    return q


def _blocks(q, nv, b):
    return q.view(q.shape[0], nv, b).permute(1, 0, 2).contiguous()


def _block_inputs(case, seed):
    n, nv, b, dt = case["n"], case["nv"], case["b"], DT[case["dt"]]
    s = {"V": _normal(seed, nv, n, b, dt=dt, salt=1), "W": _normal(seed, n, b, dt=dt, salt=2)}
    k, nc = nv * b, case["nout"] * b
    s["C"] = _normal(seed, k, nc, salt=3) / math.sqrt(k)
    if case["op"] == "combine":
        s["Out"] = torch.empty(case["nout"], n, b, dtype=dt, device="cuda")
    return s


def _expand_inputs(case, seed):
    n, nv, b = case["n"], case["nv"], case["b"]
    ptr, col = _graph(case, seed)
    V = _blocks(_basis(seed, n, nv * b), nv, b).to(DT[case["dt"]])
    return ptr, col, V


def _mlp_inputs(case, seed):
    """Features as heavy-tailed as those of a power-law graph, He-normal weights, an
    orthonormal target basis."""
    n, h, b, t = case["n"], case["h"], case["b"], case["t"]
    z = _normal(seed, n, 8, salt=1)
    f = torch.exp(1.2 * z)
    f = f / f.square().mean(0).sqrt()
    f[:, 0] = torch.log1p(torch.exp(1.5 + 1.2 * z[:, 0]))
    f[:, 7] = torch.log1p(f[:, 7])
    p = torch.cat([(_normal(seed, 8, h, salt=2) * math.sqrt(2 / 8)).flatten(), torch.zeros(h, device="cuda").double(),
                   (_normal(seed, h, h, salt=3) * math.sqrt(2 / h)).flatten(), torch.zeros(h, device="cuda").double(),
                   (_normal(seed, h, b, salt=4) * math.sqrt(1 / h)).flatten(), torch.zeros(b, device="cuda").double()])
    # unit target columns close to smooth functions of the features, as Ritz vectors are
    cols = t if case["op"] == "span" else b
    u = torch.tanh(f @ _normal(seed, 8, cols, salt=5)) + 0.5 * _normal(seed, n, cols, salt=6)
    u = torch.linalg.solve_triangular(torch.linalg.cholesky(u.T @ u).mT, u, upper=True, left=False)
    return f.float().contiguous(), p.float(), u.float().contiguous()


def prepare(case, seed):
    k = case["kind"]
    if k == "spmm":
        ptr, col = _graph(case, seed)
        X = _normal(seed, case["n"], case["b"], dt=DT[case["dt"]])
        return {"case": case, "h": _handle(case, ptr, col), "X": X, "Y": torch.empty_like(X)}
    if k == "block":
        return {"case": case, **_block_inputs(case, seed)}
    if k == "expand":
        ptr, col, V = _expand_inputs(case, seed)
        # the newest block has a buffer of its own, as spmm wants it: aligned, for any n
        return {"case": case, "h": _handle(case, ptr, col), "V": V, "x": V[-1].clone(), "W": torch.empty_like(V[0]),
                "anorm": float((ptr[1:] - ptr[:-1]).max()) ** 0.5}
    if k in ("eigs", "svds"):
        ptr, col = _graph(case, seed)
        return {"case": case, "h": _handle(case, ptr, col), "seed": int(seed) % 1000 + 1}
    F, p, U = _mlp_inputs(case, seed)
    return {"case": case, "F": F, "p": p, "U": U}


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "spmm":
        return (fe.spmm_t if c["op"] == "t" else fe.spmm)(s["h"], s["X"], s["Y"])
    if k == "block":
        if c["op"] == "gram":
            return fe.block_gram(s["V"], s["W"])
        if c["op"] == "update":
            return fe.block_update(s["V"], s["C"], s["W"], alpha=1.0, beta=0.5)
        if c["op"] == "update_gram":
            G = fe.block_update_gram(s["V"], s["C"], s["W"], alpha=1.0, beta=0.5)
            return s["W"], G
        return fe.block_combine(s["V"], s["C"], c["nout"], s["Out"])
    if k == "expand":
        W = fe.spmm(s["h"], s["x"], s["W"])
        G, R, replaced = fe.block_orth(s["V"], W, s["anorm"])
        return W, G, R, replaced
    if k == "eigs":
        ev, X, _ = fe.eigs(s["h"], c["nev"], c["b"], c["nb"], 1e-8, "LM", mode=c["mode"], seed=s["seed"],
                           max_restarts=5000)
        return ev, X
    if k == "svds":
        sv, right, left, _ = fe.svds(s["h"], c["nev"], c["b"], c["nb"], 1e-8, mode=c["mode"], seed=s["seed"],
                                     max_restarts=5000)
        return sv, right, left
    if c["op"] == "forward":
        return fe.mlp_forward(s["F"], s["p"], c["h"], c["b"])
    if c["op"] == "column":
        loss, grad = fe.mlp_loss_grad(s["F"], s["p"], c["h"], c["b"], s["U"])
    else:
        loss, grad = fe.mlp_span_loss_grad(s["F"], s["p"], c["h"], c["b"], s["U"])
    return loss, grad


# ---------------------------------------------------------------- what a pass cannot do without

def _nnz(case, directed=False):
    # measured: about 15.3 (30.6 when symmetrised) of the 16 (32) draws per vertex survive
    return int(case["n"] * (15.3 if directed else 30.6))


def _spmm_work(n, nnz, b, s):
    return 4 * nnz + 4 * (n + 1) + 2 * n * b * s, nnz * b


def work(case):
    k, n, b = case["kind"], case["n"], case["b"]
    s = 8 if case.get("dt") == "f64" else 4
    if k == "spmm":
        by, fl = _spmm_work(n, _nnz(case, case["op"] == "t"), b, s)
        return {"bytes": by, "flops": fl}
    if k == "block":
        nv, nout = case["nv"], case["nout"]
        kk = nv * b
        if case["op"] == "gram":
            return {"bytes": n * (kk + b) * s + 8 * kk * b, "flops": 2 * n * kk * b}
        if case["op"] == "update":
            return {"bytes": n * (kk + 2 * b) * s, "flops": 2 * n * kk * b}
        if case["op"] == "update_gram":
            return {"bytes": n * (kk + 2 * b) * s, "flops": 2 * n * (2 * kk + b) * b}
        return {"bytes": n * (kk + nout * b) * s, "flops": 2 * n * kk * nout * b}
    if k == "expand":
        by, fl = _spmm_work(n, _nnz(case), b, s)
        kk = case["nv"] * b
        # two Gram-Schmidt passes and Cholesky QR: the basis is read for the first coefficients,
        # for the second ones and for the last update
        return {"bytes": by + 3 * n * kk * s + 6 * n * b * s, "flops": fl + 2 * n * b * (4 * kk + 3 * b)}
    if k in ("eigs", "svds"):
        # a typical number of expansion steps: the first cycle fills the subspace, later ones
        # its free part
        nb, nev = case["nb"], case["nev"]
        directed = k == "svds"
        steps = nb * (2 if directed else 5 if nb <= 8 else 3)
        by, fl = _spmm_work(n, _nnz(case, directed), b, 8)
        ops = 2 if directed else 1
        return {"bytes": steps * (ops * by + 8 * n * b * (nb + 4)),
                "flops": steps * (ops * fl + 8 * n * b * b * nb) + 8 * n * nev}
    h = case["h"]
    macs = 8 * h + h * h + h * b
    if case["op"] == "forward":
        return {"bytes": 4 * n * (8 + b), "flops": 2 * n * macs}
    cols = case["t"] if case["op"] == "span" else b
    return {"bytes": 4 * n * (8 + cols), "flops": 6 * n * macs}


def tolerance(case):
    """About four times what the outputs were seen to differ by from the sums in FP64 (spmm, block,
    expand, mlp) on the ranges above, or from other arithmetic in the solver (eigs, svds)."""
    k = case["kind"]
    f64 = case.get("dt") == "f64"
    if k == "spmm":
        return {"rel": 8e-15, "max": 1e-12} if f64 else {"rel": 3e-7, "max": 2e-5}
    if k == "block":
        return {"rel": 1e-13, "max": 1e-12} if f64 else {"rel": 1e-5, "max": 1e-4}
    if k == "expand":
        return {"rel": 1e-13, "max": 5e-12} if f64 else {"rel": 1e-5, "max": 1e-3}
    if k in ("eigs", "svds"):
        # solves with other arithmetic that stop at the same restart agree to 1e-12; one that
        # stops a restart earlier or later has vectors off by the solver's tolerance (1e-8) over
        # the relative gap of the spectrum (1e-3 is common)
        return {"rel": 1e-5, "max": 1e-2}
    return {"rel": 2e-5, "max": 1e-3}


# ---------------------------------------------------------------- the same in plain torch, FP64

def _mul(ptr, col, X, transposed=False):
    rows = torch.repeat_interleave(torch.arange(ptr.numel() - 1, device="cuda"), ptr[1:] - ptr[:-1])
    src, dst = (rows, col) if transposed else (col, rows)
    Y = torch.zeros(ptr.numel() - 1, X.shape[1], dtype=torch.float64, device="cuda")
    for c in range(0, X.shape[1], 2):
        Y[:, c:c + 2].index_add_(0, dst, X[:, c:c + 2].double()[src])
    return Y


def _leading(apply, n, steps, count, by_size):
    """The `count` leading eigenvalues of a symmetric operator by Lanczos with full
    re-orthogonalisation."""
    Q = torch.empty(steps + 1, n, dtype=torch.float64, device="cuda")
    Q[0] = _normal(5, n)
    Q[0] /= Q[0].norm()
    T = torch.zeros(steps, steps, dtype=torch.float64)
    for j in range(steps):
        w = apply(Q[j])
        T[j, j] = float(w @ Q[j])
        for _ in range(2):
            w = w - Q[:j + 1].T @ (Q[:j + 1] @ w)
        nw = float(w.norm())
        if j + 1 < steps:
            T[j, j + 1] = T[j + 1, j] = nw
        Q[j + 1] = w / nw
    ev = torch.linalg.eigvalsh(T)
    order = torch.argsort(ev.abs() if by_size else ev, descending=True)
    return ev[order][:count].numpy()


def exact(case, seed):
    k, n, b = case["kind"], case["n"], case["b"]
    if k == "spmm":
        ptr, col = _graph(case, seed)
        return _mul(ptr, col, _normal(seed, n, b, dt=DT[case["dt"]]), case["op"] == "t")
    if k == "block":
        s = {a: x.double() for a, x in _block_inputs(case, seed).items()}
        V = s["V"].permute(1, 0, 2).reshape(n, -1)
        if case["op"] == "gram":
            return V.T @ s["W"]
        if case["op"] == "combine":
            return _blocks(V @ s["C"], case["nout"], b)
        W = 0.5 * s["W"] + V @ s["C"]
        return W if case["op"] == "update" else (W, torch.cat([V, W], 1).T @ W)
    if k == "expand":
        ptr, col, V = _expand_inputs(case, seed)
        W = _mul(ptr, col, V[-1])
        V = V.permute(1, 0, 2).reshape(n, -1).double()
        G = torch.zeros(V.shape[1], b, dtype=torch.float64, device="cuda")
        for _ in range(2):
            g = V.T @ W
            W, G = W - V @ g, G + g
        R = torch.eye(b, dtype=torch.float64, device="cuda")
        for _ in range(2):
            r = torch.linalg.cholesky(W.T @ W).mT
            W, R = torch.linalg.solve_triangular(r, W, upper=True, left=False), r @ R
        return W, G, R, None
    if k in ("eigs", "svds"):
        ptr, col = _graph(case, seed)
        A = torch.sparse_csr_tensor(ptr, col, torch.ones(col.numel(), dtype=torch.float64, device="cuda"), (n, n))
        if k == "eigs":
            steps = min(n - 1, 500 if case["nev"] <= 8 else 700)
            return _leading(lambda x: A @ x, n, steps, case["nev"], True), None
        rows = torch.repeat_interleave(torch.arange(n, device="cuda"), ptr[1:] - ptr[:-1])
        key = torch.sort(col * n + rows).values
        tptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        tptr[1:] = torch.cumsum(torch.bincount(col, minlength=n), 0)
        At = torch.sparse_csr_tensor(tptr, key % n, torch.ones(col.numel(), dtype=torch.float64, device="cuda"), (n, n))
        ev = _leading(lambda x: At @ (A @ x), n, min(n - 1, 300), case["nev"], False)
        return np.sqrt(ev), None, None
    F, p, U = (x.double() for x in _mlp_inputs(case, seed))
    h = case["h"]
    p = p.detach().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(p, [8 * h, h, h * h, h, h * b, b])
    Z = torch.relu(torch.relu(F @ w1.view(8, h) + b1) @ w2.view(h, h) + b2) @ w3.view(h, b) + b3
    if case["op"] == "forward":
        return Z.detach()
    S = U.T @ Z
    if case["op"] == "column":
        loss = (1 - torch.diagonal(S).square() / Z.square().sum(0)).sum()
    else:
        loss = b - torch.trace(torch.linalg.solve(Z.T @ Z, S.T @ S))
    (g,) = torch.autograd.grad(loss, p)
    return float(loss.detach()), g
