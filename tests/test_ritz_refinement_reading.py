"""CPU pin of the Rayleigh-Ritz up to subspace 160, independent of the GPU code: FP32 Jacobi sweeps whose
result is refined by FP64 matrix products (the treatment of the basis's error follows Ogita & Aishima,
Japan J. Indust. Appl. Math. 35, 2018) give eigenpairs to FP64 accuracy.

Restated, with FP32 where the kernel has FP32 (the sweeps run pair by pair here, in parallel steps
there): Q, diagonal d and remainder N start as I, diag T and T's off-diagonal.  An iteration
  * forms E, the rotation relative to I that diagonalises d + N: Jacobi sweeps in FP32 on N, d and E with
    the diagonal as two floats, leaving alone entries below `skip`, and those below tau (what N itself is
    uncertain by) whose angle would not be tiny; or, once every angle is below 1e-8, N_ij / (d_j - d_i);
  * Q <- Q + Q (R / 2 + E), R = I - Q^T Q (the first time Q = I + E), G = Q^T Q, S = Q^T T Q in FP64;
  * d <- diag S + R_ii d_i, N_ij <- S_ij + R_ij (d_i + d_j) / 2, rounded to FP32.
It ends after a first-order E with |R| <= 1e-8."""
import numpy as np
import pytest

F = np.float32
TINY = F(1e-8)


def _rotation(n, gap):
    """(cos - 1, sin, tan) of the angle that zeroes n for the diagonal difference gap, FP32."""
    g, h = abs(gap), F(2) * n
    w = F(np.hypot(F(g), F(h)))
    if w == 0:
        return F(0), F(0), F(0)
    c = F(np.sqrt(F(0.5) + F(0.5) * F(g / w)))
    s = F(np.copysign(F(0.5), gap) * h / w / c)
    return F(-s * s / (F(1) + c)), s, F(s / c)


def _sweeps(N, d, tau, skip, cap, first, fro, use_tau=True):
    """FP32 Jacobi sweeps on d + N; (E, d) with the diagonal as two floats, E relative to I."""
    m = len(d)
    N = N.copy()
    hi, lo = d.astype(F), (d - d.astype(F).astype(float)).astype(F)
    E = np.zeros((m, m), F)
    for _ in range(cap):
        pivots, top = 0.0, F(0)
        for p in range(m):
            for q in range(p + 1, m):
                n = N[p, q]
                gap = F(F(hi[q] - hi[p]) + F(lo[q] - lo[p]))
                if not (abs(n) > skip and (not use_tau or abs(n) > tau or abs(n) <= TINY * abs(gap))):
                    continue
                cm, s, t = _rotation(n, gap)
                pivots += float(n) ** 2
                top = max(top, abs(t))
                for k in (p, q):                       # the diagonal, as an unevaluated sum
                    x = F(lo[k] + (F(-t) * n if k == p else t * n))
                    hi[k], lo[k] = F(hi[k] + x), F(x - F(F(hi[k] + x) - hi[k]))
                rows = N[[p, q], :].copy()
                N[p, :] = rows[0] + (cm * rows[0] - s * rows[1])
                N[q, :] = rows[1] + (cm * rows[1] + s * rows[0])
                cols = N[:, [p, q]].copy()
                N[:, p] = cols[:, 0] + (cm * cols[:, 0] - s * cols[:, 1])
                N[:, q] = cols[:, 1] + (cm * cols[:, 1] + s * cols[:, 0])
                N[p, q] = N[q, p] = F(0)
                N[p, p] = N[q, q] = F(0)
                e = E[:, [p, q]].copy()
                vp, vq = e[:, 0].copy(), e[:, 1].copy()
                vp[p] += F(1)
                vq[q] += F(1)
                E[:, p] = e[:, 0] + (cm * vp - s * vq)
                E[:, q] = e[:, 1] + (cm * vq + s * vp)
        if (pivots <= 1e-8 * fro ** 2) if first else (top <= F(1e-4)):
            break
    return E.astype(float), hi.astype(float) + lo.astype(float)


def ritz(T, tol=1e-15, treat_basis=True, use_tau=True):
    """(theta, Q, iterations) of the symmetric T."""
    m = len(T)
    fro = float(np.linalg.norm(T))
    Q, d = np.eye(m), np.diag(T).copy()
    N = (T - np.diag(d)).astype(F)
    R = np.zeros((m, m))
    for it in range(9):
        rmax = F(np.abs(R).max())
        tau = F(tol * fro) if it == 0 else max(F(tol * fro), F(0.5) * m * rmax * rmax * F(np.abs(d).max()))
        gap = np.abs(d[None, :] - d[:, None])
        off = ~np.eye(m, dtype=bool) & (N != 0)
        aN = np.abs(N)
        seen = off & ((aN > tau) | (aN <= float(TINY) * gap))
        with np.errstate(divide="ignore", invalid="ignore"):
            emax = np.where(gap > 0, aN / gap, 1.0)[seen].max() if seen.any() else 0.0
        first_order = it > 0 and emax <= TINY
        if first_order:
            g = (d[None, :] - d[:, None]).astype(F)
            take = off & (aN <= TINY * np.abs(g)) & (g != 0)
            E = np.where(take, N / np.where(g == 0, F(1), g), F(0)).astype(float)
        else:
            nu = float(aN.max())
            skip = F(max(2e-8 * fro if it == 0 else 1e-7 * nu, 1e-17 * fro))
            E, d = _sweeps(N, d, tau, skip, 15 if it == 0 else 6, it == 0, fro, use_tau)
        Q = np.eye(m) + E if it == 0 else Q + Q @ ((R / 2 if treat_basis else 0.0) + E)
        if first_order and rmax <= TINY:
            return d, Q, it
        G = Q.T @ Q
        S = Q.T @ (T @ Q)
        R = np.eye(m) - G
        prev = d
        d = np.diag(S) + np.diag(R) * prev
        N = (S + 0.5 * R * (prev[None, :] + prev[:, None])).astype(F)
        N = np.triu(N, 1)
        N = N + N.T                                    # one triangle is computed, the other mirrored
    return d, Q, 9


def _matrices():
    r = np.random.default_rng(0)
    m = 24
    X = r.standard_normal((m, m))
    yield "normal", (X + X.T) / 2
    U, _ = np.linalg.qr(r.standard_normal((m, m)))
    yield "repeated", (U * np.repeat([8.0, 6.0, 4.0, -6.0], 6)) @ U.T
    yield "close", (U * (1.0 + 1e-9 * np.arange(m))) @ U.T
    yield "one large", (U * np.concatenate([[1e3], r.standard_normal(m - 1)])) @ U.T
    A = np.diag(r.standard_normal(m))
    A[-4:, :] = 0.3 * r.standard_normal((4, m))           # as after a restart: a diagonal and a border
    yield "restarted", (A + A.T) / 2
    yield "diagonal", np.diag(np.arange(m, dtype=float))


@pytest.mark.parametrize("name,T", list(_matrices()), ids=[n for n, _ in _matrices()])
def test_refined_pairs_reach_fp64(name, T):
    """Residuals and orthonormality to a few FP64 roundings of products of 24 terms, eigenvalues as
    numpy's, in at most three iterations after the FP32 one."""
    T = (T + T.T) / 2
    d, Q, it = ritz(T)
    scale = np.linalg.norm(T, 2)
    assert it <= 3
    assert np.abs(Q.T @ Q - np.eye(len(T))).max() < 2e-15
    assert np.abs(T @ Q - Q * d).max() < 1e-14 * scale
    assert np.abs(np.sort(d) - np.linalg.eigvalsh(T)).max() < 1e-14 * scale


def test_fp32_sweeps_alone_do_not():
    """The pin is sensitive: the first iteration's vectors are good to FP32 only, and without the
    correction by the basis's own error R they stay unorthogonal."""
    T = dict(_matrices())["normal"]
    fro = float(np.linalg.norm(T))
    E, _ = _sweeps((T - np.diag(np.diag(T))).astype(F), np.diag(T).copy(), F(1e-15 * fro), F(2e-8 * fro), 15, True, fro)
    Q = np.eye(len(T)) + E
    assert 1e-8 < np.abs(Q.T @ Q - np.eye(len(T))).max() < 1e-5
    _, Q, _ = ritz(T, treat_basis=False)
    assert np.abs(Q.T @ Q - np.eye(len(T))).max() > 1e-9
