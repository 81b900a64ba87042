"""GPU parity of the Table 1 block operations and the re-orthogonalisation step against the
oracle (numpy FP64 on the same inputs).

Bounds: a k-term FP64 sum errs by at most ~k u |terms|; the kernels sum <= 64 rows per lane
and then combine in FP64, so FP64 results are held to 1e-13 and FP32 ones to 1e-5 of the
absolute-value product (|V|^T |W|, |V| |C| + |beta W|).
"""
import numpy as np
import pytest

import graphgen
import paper_1602_01421_gb300 as fe
from oracle import bks, blockops, rng
from tests.gpu_util import to_dev, torch

pytestmark = pytest.mark.gpu
NP = {"f32": np.float32, "f64": np.float64}
TOL = {"f32": 1e-5, "f64": 1e-13}


def _blocks(nv, n, bv, seed, dtype):
    return graphgen.normal_block(nv * n, bv, seed=seed, dtype=dtype).reshape(nv, n, bv)


def _as_tall(V):
    nv, n, bv = V.shape
    return np.concatenate([V[j] for j in range(nv)], axis=1).astype(np.float64)  # n x nv*bv


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,nv,bv,bw", [(1, 1, 1, 1), (1000, 1, 4, 4), (5003, 9, 4, 4),
                                        (70001, 17, 4, 4), (33000, 5, 8, 8), (20000, 3, 16, 16),
                                        (12345, 2, 2, 8), (4099, 32, 1, 2), (9001, 128, 4, 4)])
def test_gram_parity(prec, n, nv, bv, bw):
    V = _blocks(nv, n, bv, 1, NP[prec])
    W = graphgen.normal_block(n, bw, seed=2, dtype=NP[prec])
    G = fe.block_gram(to_dev(V), to_dev(W), alpha=0.5).cpu().numpy()
    Vt, W64 = _as_tall(V), W.astype(np.float64)
    ref = blockops.mv_trans_mv(0.5, Vt, W64)
    bound = TOL[prec] * 0.5 * (np.abs(Vt).T @ np.abs(W64)) + 1e-300
    assert np.all(np.abs(G - ref) <= bound)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,nv,bv,bw", [(1, 1, 1, 1), (5003, 9, 4, 4), (70001, 16, 4, 4),
                                        (33000, 8, 8, 8), (2000, 2, 16, 16), (999, 0, 4, 4),
                                        (9001, 128, 4, 4)])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (0.25, 0.0), (2.0, -3.0)])
def test_update_parity(prec, n, nv, bv, bw, alpha, beta):
    t = torch()
    V = _blocks(max(nv, 1), n, bv, 3, NP[prec])[:nv] if nv else None
    C = np.random.default_rng(4).standard_normal((max(nv, 1) * bv, bw))[: nv * bv]
    W = graphgen.normal_block(n, bw, seed=5, dtype=NP[prec])
    Wd = to_dev(W)
    fe.block_update(None if V is None else to_dev(V), to_dev(C), Wd, alpha, beta)
    got = Wd.cpu().numpy().astype(np.float64)
    W64 = W.astype(np.float64)
    if nv:
        Vt = _as_tall(V)
        ref = blockops.mv_times_mat_add_mv(alpha, Vt, C, beta, W64)
        mag = np.abs(alpha) * (np.abs(Vt) @ np.abs(C)) + np.abs(beta * W64)
    else:
        ref = blockops.mv_scale1(beta, W64)
        mag = np.abs(beta * W64)
    k = nv * bv + bw + 2
    rel = {"f32": 6e-8, "f64": 1.2e-16}[prec] * k * 2
    assert np.all(np.abs(got - ref) <= rel * mag + 1e-300)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,nv,b", [(1, 0, 1), (999, 0, 4), (5003, 3, 4), (70001, 7, 4),
                                    (4099, 8, 4), (33000, 12, 2), (20000, 17, 4), (7777, 5, 8),
                                    (3000, 15, 1), (6001, 128, 4)])
@pytest.mark.parametrize("alpha,beta", [(-1.0, 1.0), (0.5, -2.0)])
def test_update_gram_parity(prec, n, nv, b, alpha, beta):
    """fe_block_update_gram = op1 then op3 on the updated block (oracle: the two Table 1
    operations one after the other, FP64).  Shapes span one warp per tile (<= 16 tiles: block
    of 32 x tiles threads), the per-range reduction (17 blocks), ragged row tails."""
    V = _blocks(max(nv, 1), n, b, 6, NP[prec])[:nv] if nv else None
    C = np.random.default_rng(7).standard_normal((max(nv, 1) * b, b))[: nv * b]
    W = graphgen.normal_block(n, b, seed=8, dtype=NP[prec])
    Wd = to_dev(W)
    G = fe.block_update_gram(None if V is None else to_dev(V), to_dev(C), Wd, alpha, beta)
    got_w = Wd.cpu().numpy().astype(np.float64)
    got_g = G.cpu().numpy()
    W64 = W.astype(np.float64)
    if nv:
        Vt = _as_tall(V)
        ref_w = blockops.mv_times_mat_add_mv(alpha, Vt, C, beta, W64)
        mag = np.abs(alpha) * (np.abs(Vt) @ np.abs(C)) + np.abs(beta * W64)
    else:
        Vt = np.zeros((n, 0))
        ref_w = blockops.mv_scale1(beta, W64)
        mag = np.abs(beta * W64)
    k = nv * b + b + 2
    rel = {"f32": 6e-8, "f64": 1.2e-16}[prec] * k * 2
    assert np.all(np.abs(got_w - ref_w) <= rel * mag + 1e-300)
    # Gram of [V; W_new] against W_new, from the kernel's own W_new (the update's rounding is
    # checked above): bound by |[V W]|^T |W| like the Gram test
    VW = np.concatenate([Vt, got_w], axis=1)
    ref_g = blockops.mv_trans_mv(1.0, VW, got_w)
    bound = TOL[prec] * (np.abs(VW).T @ np.abs(got_w)) + 1e-300
    assert got_g.shape == ((nv + 1) * b, b)
    assert np.all(np.abs(got_g - ref_g) <= bound)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_random_normal_matches_oracle_generator(prec):
    t = torch()
    X = fe.random_normal(10007, 4, dtype=t.float32 if prec == "f32" else t.float64, seed=7,
                         stream=4, offset=123).cpu().numpy()
    ref = rng.normal_block(10007, 4, seed=7, stream=4, offset=123)
    assert np.allclose(X, ref, rtol={"f32": 1e-6, "f64": 1e-13}[prec], atol={"f32": 1e-6, "f64": 1e-13}[prec])


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n,nv,b", [(20000, 0, 4), (20000, 3, 4), (50001, 7, 8), (9000, 2, 16),
                                    (3000, 12, 1)])
def test_orth_matches_oracle(prec, n, nv, b):
    """CGS2 + CholQR2 (Section 3.1 re-orthogonalisation) vs oracle.bks.orth_block."""
    r = np.random.default_rng(nv * 100 + b)
    Vt, _ = np.linalg.qr(r.standard_normal((n, max(nv, 1) * b)))
    Vt = Vt[:, : nv * b]
    V = np.stack([Vt[:, j * b:(j + 1) * b] for j in range(nv)]) if nv else None
    W = r.standard_normal((n, b)) + (Vt @ r.standard_normal((nv * b, b)) if nv else 0.0)
    Wd = to_dev(W.astype(NP[prec]))
    G, R, rep = fe.block_orth(None if V is None else to_dev(V.astype(NP[prec])), Wd, anorm=10.0)
    Q = Wd.cpu().numpy().astype(np.float64)
    G, R = G.cpu().numpy(), R.cpu().numpy()
    W64 = W.astype(NP[prec]).astype(np.float64)
    Vq = Vt.astype(NP[prec]).astype(np.float64)
    Qo, Go, Ro = bks.orth_block(Vq if nv else np.zeros((n, 0)), W64, 10.0, 1,
                                {"counter": 0, "replacements": 0})
    tol = {"f32": 2e-5, "f64": 1e-11}[prec]
    assert rep == 0
    assert np.allclose(R, Ro, rtol=tol, atol=tol * np.abs(Ro).max())
    if nv:
        assert np.allclose(G, Go, rtol=tol, atol=tol * np.abs(Go).max())
    assert np.abs(Q.T @ Q - np.eye(b)).max() < {"f32": 1e-5, "f64": 1e-13}[prec]
    if nv:
        assert np.abs(Vq.T @ Q).max() < {"f32": 1e-5, "f64": 1e-13}[prec]
    recon = (Vq @ G if nv else 0.0) + Q @ R
    assert np.abs(recon - W64).max() < {"f32": 1e-4, "f64": 1e-11}[prec] * np.abs(W64).max()


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_orth_breakdown_replaces_columns(prec):
    """W with two columns inside span(V) and one duplicate: three random replacements,
    R[i][i] = 0 for them, output still orthonormal and orthogonal to V."""
    n, b, nv = 4000, 4, 2
    r = np.random.default_rng(3)
    Vt, _ = np.linalg.qr(r.standard_normal((n, nv * b)))
    V = np.stack([Vt[:, j * b:(j + 1) * b] for j in range(nv)])
    W = np.empty((n, b))
    W[:, 0] = r.standard_normal(n)
    W[:, 1] = Vt @ r.standard_normal(nv * b)
    W[:, 2] = 2.0 * W[:, 0]
    W[:, 3] = Vt @ r.standard_normal(nv * b)
    Wd = to_dev(W.astype(NP[prec]))
    G, R, rep = fe.block_orth(to_dev(V.astype(NP[prec])), Wd, anorm=100.0, seed=5)
    Q = Wd.cpu().numpy().astype(np.float64)
    R = R.cpu().numpy()
    if prec == "f64":
        assert rep == 3
        assert R[1, 1] == 0.0 and R[2, 2] == 0.0 and R[3, 3] == 0.0
    else:
        # FP32 remainders of dependent columns are rounding noise (~1e-7 |w|), far above the
        # 1e-12 ||A|| breakdown level: they are kept as (random) directions, R[i][i] tiny
        assert abs(R[1, 1]) < 1e-5 * abs(R[0, 0]) and abs(R[3, 3]) < 1e-5 * abs(R[0, 0])
    assert np.abs(Q.T @ Q - np.eye(b)).max() < {"f32": 1e-5, "f64": 1e-12}[prec]
    assert np.abs(Vt.T @ Q).max() < {"f32": 1e-5, "f64": 1e-12}[prec]
    recon = Vt @ G.cpu().numpy() + Q @ R
    assert np.abs(recon - W).max() < {"f32": 1e-4, "f64": 1e-10}[prec] * np.abs(W).max()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nv,nout,bv", [(128, 64, 4), (64, 100, 4), (32, 128, 2)])
def test_combine_many_blocks_matches_oracle(prec, nv, nout, bv):
    """The restart product with large subspaces (up to 128 input and output blocks, several
    launches of the coefficient-tiled FMA kernel) against the oracle's op1."""
    n = 3001
    V = _blocks(nv, n, bv, 7, NP[prec])
    Y = np.random.default_rng(8).standard_normal((nv * bv, nout * bv))
    out = fe.block_combine(to_dev(V), to_dev(Y), nout, engine="fma").cpu().numpy()
    got = np.concatenate([out[o] for o in range(nout)], axis=1).astype(np.float64)
    Vt = _as_tall(V)
    ref = Vt @ Y
    rel = {"f32": 6e-8, "f64": 1.2e-16}[prec] * (nv * bv + 2) * 2
    assert np.all(np.abs(got - ref) <= rel * (np.abs(Vt) @ np.abs(Y)) + 1e-300)


@pytest.mark.parametrize("b", [1, 2, 4])
@pytest.mark.parametrize("n", [1, 31, 255, 257, 8193, 320 * 256, 320 * 256 + 1])
def test_orth_partial_sums(n, b):
    """W^T W of the last pass, added by the factorisation itself from 1 to 320 partial sums and by a
    kernel of its own beyond: W's columns are orthonormal to 1e-13 and R is the Cholesky factor to
    1e-11 (conditions below 1e2 times the FP64 rounding of sums of n terms)."""
    r = np.random.default_rng(n + b)
    b = min(b, n)   # one row: one column
    W = r.standard_normal((n, b)) + np.eye(n, b) * 4.0
    Wd = to_dev(W)
    G, R, rep = fe.block_orth(None, Wd, anorm=10.0)
    Q, want = Wd.cpu().numpy(), np.linalg.cholesky(W.T @ W).T
    assert rep == 0
    assert np.abs(R.cpu().numpy() - want).max() < 1e-11 * np.abs(want).max()
    assert np.abs(Q.T @ Q - np.eye(b)).max() < 1e-13


@pytest.mark.parametrize("n,nv,b,scale", [(5000, 3, 2, 1.0), (5000, 2, 16, 1.0), (2000, 5, 1, 1.0), (4000, 2, 4, 1e-100),
                                          (4000, 2, 4, 1e120), (4000, 2, 4, 1e-145), (4000, 0, 8, 1e145)])
def test_orth_factorisation_widths_and_scales(n, nv, b, scale):
    """The one-warp Cholesky factorisation at every width, and with Gram diagonals (scale^2 n) inside
    and outside the range of its Newton-corrected square roots.  Everything scales with W, so the
    bounds are those of scale 1: R is the Cholesky factor of the projected W to 1e-11 (its
    condition, below 1e2, times FP64 rounding of sums of n terms)."""
    r = np.random.default_rng(n + b)
    Vt, _ = np.linalg.qr(r.standard_normal((n, max(nv, 1) * b)))
    Vt = Vt[:, : nv * b]
    W = r.standard_normal((n, b))
    Wd = to_dev(W * scale)
    V = to_dev(np.stack([Vt[:, j * b:(j + 1) * b] for j in range(nv)])) if nv else None
    G, R, rep = fe.block_orth(V, Wd, anorm=10.0 * scale)
    Q, R = Wd.cpu().numpy(), R.cpu().numpy() / scale
    P = W - Vt @ (Vt.T @ W) if nv else W
    want = np.linalg.cholesky(P.T @ P).T
    assert rep == 0
    assert np.abs(R - want).max() < 1e-11 * np.abs(want).max()
    assert np.abs(Q.T @ Q - np.eye(b)).max() < 1e-13
    if nv:
        assert np.abs(G.cpu().numpy() / scale - Vt.T @ W).max() < 1e-11 * np.abs(want).max()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("b", [1, 2, 4, 8])
@pytest.mark.parametrize("n,nv", [(1, 1), (31, 2), (33, 3), (255, 4), (256, 5), (257, 7), (70001, 8), (3001, 9), (5000, 15),
                                  (5001, 16), (4099, 17), (4100, 31), (2000, 32), (2000, 33)])
def test_row_sweeps(prec, b, n, nv):
    """Gram and update + Gram at the edges of the row sweeps: every number of lanes per row (1, 2, 4,
    8, the next one falling back to the tile kernels), one row, ragged last rows, more rows than a
    grid holds at once.  Bounds: sums of k products in FP32 (FP64) have errors of a few
    sqrt(k) 2^-24 (2^-53) of |V|^T|W|; 32 times that rate allowed for k = n."""
    r = np.random.default_rng(1000 * b + nv)
    V = r.standard_normal((nv, n, b)).astype(NP[prec])
    W = r.standard_normal((n, b)).astype(NP[prec])
    C = r.standard_normal((nv * b, b)) / np.sqrt(nv * b)
    V64 = np.concatenate([v.astype(np.float64) for v in V], axis=1)
    u = {"f32": 2.0 ** -24, "f64": 2.0 ** -53}[prec]
    G = fe.block_gram(to_dev(V), to_dev(W), alpha=-0.5, engine="fma").cpu().numpy()
    want, mag = -0.5 * (V64.T @ W.astype(np.float64)), 0.5 * (np.abs(V64).T @ np.abs(W).astype(np.float64))
    assert np.all(np.abs(G - want) <= 32 * u * mag + 1e-300)
    Wd = to_dev(W)
    G = fe.block_update_gram(to_dev(V), to_dev(C), Wd, alpha=1.0, beta=0.5).cpu().numpy()
    Wn = 0.5 * W.astype(np.float64) + V64 @ C
    magw = 0.5 * np.abs(W).astype(np.float64) + np.abs(V64) @ np.abs(C)
    got = Wd.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - Wn) <= (nv * b + 8) * u * magw)
    X = np.concatenate([V64, got], axis=1)
    assert np.all(np.abs(G - X.T @ got) <= 32 * u * (np.abs(X).T @ np.abs(got)) + 1e-300)


def test_row_sweep_large_sums_and_infinities():
    """FP32 Grams whose sums leave FP32's range are finite in G (FP64), and an infinite entry makes the
    entries it enters infinite, not NaN."""
    n = 4096
    V = np.full((2, n, 4), 3e18, np.float32)
    W = np.full((n, 4), 3e19, np.float32)
    G = fe.block_gram(to_dev(V), to_dev(W)).cpu().numpy()
    want = n * float(np.float32(3e18)) * float(np.float32(3e19))
    assert np.allclose(G, want, rtol=1e-6)
    V[1, 77, 2] = np.inf
    G = fe.block_gram(to_dev(V), to_dev(W)).cpu().numpy()
    assert np.all(np.isposinf(G[6])) and np.isfinite(G[:6]).all() and np.isfinite(G[7]).all()


@pytest.mark.parametrize("n", [1, 33, 257, 5001])
def test_row_sweep_infinite_coefficients(n):
    """An infinite coefficient makes W's column infinite and with it the entries of G that W enters: rows
    past the end of a ragged range (0 times infinity) do not turn them into NaN."""
    r = np.random.default_rng(n)
    V = r.random((3, n, 4)).astype(np.float32) + 0.5
    W = r.random((n, 4)).astype(np.float32) + 0.5
    C = r.random((12, 4))
    C[5, 2] = np.inf
    Wd = to_dev(W)
    G = fe.block_update_gram(to_dev(V), to_dev(C), Wd, alpha=1.0, beta=0.5).cpu().numpy()
    got = Wd.cpu().numpy()
    other = [0, 1, 3]
    assert np.all(np.isposinf(got[:, 2])) and np.isfinite(got[:, other]).all()
    assert np.all(np.isposinf(G[:, 2])) and np.all(np.isposinf(G[14, :]))
    assert np.isfinite(G[np.ix_([i for i in range(16) if i != 14], other)]).all()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -62, 2.0 ** 56])
@pytest.mark.parametrize("b,nv,n", [(8, 8, 1 << 20), (8, 15, 600011), (8, 2, 1 << 21), (4, 31, 1 << 21), (4, 16, 1 << 20),
                                    (2, 20, 1 << 21), (2, 60, 600011), (1, 20, 1 << 21), (1, 60, 1 << 20)])
def test_row_sweep_long_sums(b, nv, n, scale):
    """FP32 sums of the shapes that a launch does not keep in one accumulator run over 8 rows (update +
    Gram of b = 8 or more than 16 tiles), 16 (Gram of b = 8, more than 4 blocks) or 32 (more than 16 blocks
    of 4): whatever n, the error is at most that many units of 2^-24, and one for the rest, which is as
    good as FP64.  The two constants' products round the same way in every addition: a sum of 200 is
    48 units off.  Also with products near the smallest normal number (2^-122) and with sums that leave
    FP32's range (2^113 each)."""
    t = __import__("torch")
    v, w = np.float32(1.4888460636138916), np.float32(1.9886953830718994)
    V = t.full((nv, n, b), float(v) * scale, dtype=t.float32, device="cuda")
    W = t.full((n, b), float(w) * scale, dtype=t.float32, device="cuda")
    vw, ww = n * float(v) * float(w) * scale ** 2, n * float(w) ** 2 * scale ** 2
    u = 2.0 ** -24
    G = fe.block_update_gram(V, t.zeros(nv * b, b, dtype=t.float64, device="cuda"), W, alpha=1.0, beta=1.0).cpu().numpy()
    assert np.abs(G[:nv * b] / vw - 1).max() <= 9 * u and np.abs(G[nv * b:] / ww - 1).max() <= 9 * u
    assert np.array_equal(G[nv * b:], G[nv * b:].T)
    run = 16 if b == 8 and nv > 4 else 32 if b == 4 and nv > 16 else 0
    if run:
        G = fe.block_gram(V, W, engine="fma").cpu().numpy()
        assert np.abs(G / vw - 1).max() <= (run + 1) * u


@pytest.mark.parametrize("b,nv,n", [(2, 20, 1 << 17), (2, 20, (1 << 17) + 1), (2, 24, 140001), (2, 25, 140001), (1, 17, (1 << 25) // 17),
                                    (1, 17, (1 << 25) // 17 + 1), (8, 3, 65535), (8, 3, 65536), (8, 5, 70001), (8, 7, 70001),
                                    (4, 19, 70001), (4, 20, 70001)])
def test_fp64_kernel_choice(b, nv, n):
    """Both sides of the rules that choose between the row sweeps and the tile kernels in FP64: Gram and
    update + Gram against torch's FP64 products of the same data.  Bounds: twice those of test_row_sweeps,
    since both sides round."""
    t = __import__("torch")
    g = t.Generator(device="cuda").manual_seed(n + nv)
    V = t.randn(nv, n, b, generator=g, device="cuda", dtype=t.float64)
    W = t.randn(n, b, generator=g, device="cuda", dtype=t.float64)
    C = t.randn(nv * b, b, generator=g, device="cuda", dtype=t.float64) / (nv * b) ** 0.5
    A = V.permute(1, 0, 2).reshape(n, -1)
    u = 2.0 ** -53
    G = fe.block_gram(V, W, engine="fma")
    assert ((G - A.T @ W).abs() <= 64 * u * (A.abs().T @ W.abs())).all()
    want = 0.5 * W + A @ C
    mag = 0.5 * W.abs() + A.abs() @ C.abs()
    G = fe.block_update_gram(V, C, W, alpha=1.0, beta=0.5)
    assert ((W - want).abs() <= 2 * (nv * b + 8) * u * mag).all()
    A = t.cat([A, W], 1)
    assert ((G - A.T @ W).abs() <= 64 * u * (A.abs().T @ W.abs())).all()
