"""FP64 solves of one to four columns (one launch per level) and the coupling
matrices' FP64 products: leaf sizes and ranks around their tiles, trees with one and
with many projection chunks per node, strided columns, bad operators (GPU)."""
import numpy as np
import pytest
import torch

from oracle.hodlr import RecursiveHODLR
from synth import HodlrShape, gaussian_rhs, synthetic_hodlr, to_math

pytestmark = pytest.mark.gpu


def case(m, L, r, k, seed):
    N = m << L
    D, U, V, g = synthetic_hodlr(HodlrShape(N, L, r), 4.0, seed)
    B = gaussian_rhs(N, k, g)
    return to_math(D, U, V, B), tuple(t.to("cuda") for t in (D, U, V, B))


# solutions of these operators (condition numbers of a few tens) agree with the
# oracle's to a few hundred roundings; more than eight chunks per child from 12 levels
# of 16 rows (chunks of 128) and from 2^16 rows (chunks of 256) on
@pytest.mark.parametrize("m,L,r,k", [
    (1, 1, 1, 1), (5, 3, 2, 3), (16, 11, 4, 1), (31, 4, 31, 2), (33, 3, 9, 4), (64, 6, 16, 1), (64, 4, 33, 3),
    (100, 4, 21, 4), (127, 3, 64, 2), (128, 9, 8, 2), (129, 3, 47, 1), (200, 8, 6, 3), (255, 2, 32, 4),
    (256, 3, 64, 4), (256, 8, 17, 1)])
def test_small_solves(cuda_lib, m, L, r, k):
    hb = cuda_lib
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=m + r)
    rec = RecursiveHODLR(Dm, Um, Vm, L)
    F = hb.hodlr_factor(D, U, V, L, r, "fp64")
    for got, ref in ((hb.hodlr_solve(F, B.clone()), rec.solve(Bm)),
                     (hb.hodlr_solve_adjoint(F, B.clone()), rec.solve_adjoint(Bm))):
        np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
    s, la = hb.hodlr_logdet(F)
    so, lao = rec.slogdet()
    assert s == so and abs(la - lao) <= 1e-12 * max(1.0, abs(lao))


def test_small_solve_strided(cuda_lib):
    hb = cuda_lib
    m, L, r, k = 60, 5, 12, 3
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=2)
    N = m << L
    buf = torch.full((k, N + 5), 7.0, dtype=torch.float64, device="cuda").T
    X = buf[1:1 + N]
    X.copy_(B)
    hb.hodlr_solve(hb.hodlr_factor(D, U, V, L, r, "fp64"), X)
    ref = RecursiveHODLR(Dm, Um, Vm, L).solve(Bm)
    np.testing.assert_allclose(X.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
    assert (buf[:1] == 7).all() and (buf[1 + N:] == 7).all()


@pytest.mark.parametrize("r", [1, 7, 16, 32, 33, 64])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_coupling_pivots(cuda_lib, r, prec):
    """Coupling matrices whose Schur complement needs row exchanges: D = I and bases
    that make T_a T_b = I + a shuffled diagonal, so S is a signed permutation."""
    hb = cuda_lib
    m, L = 64, 1
    rng = np.random.default_rng(r)
    perm, sign = rng.permutation(r), rng.choice([-1.0, 1.0], r)
    S = np.zeros((r, r))
    S[np.arange(r), perm] = sign * rng.uniform(0.5, 2.0, r)
    N = 2 * m
    U, V = np.zeros((N, r)), np.zeros((N, r))
    U[:r], V[:r] = np.eye(r), np.eye(r)              # T_a = I
    U[m:m + r], V[m:m + r] = np.eye(r) - S, np.eye(r)  # T_b = I - S, so I - T_a T_b = S
    D = np.stack([np.eye(m)] * 2)
    B = rng.standard_normal((N, 2))
    Dt = torch.from_numpy(D.copy()).cuda().transpose(1, 2).contiguous().transpose(1, 2)
    Ut, Vt, Bt = (torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T for a in (U, V, B))
    F = hb.hodlr_factor(Dt, Ut, Vt, L, r, prec)
    rec = RecursiveHODLR(D, U, V, L)
    tol = 1e-12 if prec == "fp64" else 1e-4
    x = hb.hodlr_solve(F, Bt.clone()).cpu().numpy()
    ref = rec.solve(B)
    np.testing.assert_allclose(x, ref, rtol=0, atol=tol * np.abs(ref).max())
    s, la = hb.hodlr_logdet(F)
    so, lao = rec.slogdet()
    assert s == so and abs(la - lao) <= tol * max(1.0, abs(lao))


@pytest.mark.parametrize("r", [4, 40])
def test_singular_coupling(cuda_lib, r):
    hb = cuda_lib
    m, L = 64, 1
    N = 2 * m
    U = np.zeros((N, r))
    U[:r], U[m:m + r] = np.eye(r), np.eye(r)  # T_a = T_b = I: S = 0
    D = torch.eye(m, dtype=torch.float64, device="cuda").repeat(2, 1, 1).transpose(1, 2)
    Ut = torch.from_numpy(np.ascontiguousarray(U.T)).cuda().T
    with pytest.raises(hb.HodlrError) as e:
        hb.hodlr_logdet(hb.hodlr_factor(D, Ut, Ut.T.clone().T, L, r, "fp64"))
    assert e.value.code == hb.HODLR_ERR_SINGULAR_COUPLING


@pytest.mark.parametrize("m,L,r", [(64, 4, 8), (256, 3, 64), (100, 7, 21)])
def test_solve_workspace_serves_fewer_columns(cuda_lib, m, L, r):
    """A workspace sized for some number of columns is large enough for fewer."""
    hb = cuda_lib
    _, (D, U, V, _) = case(m, L, r, 1, seed=1)
    for prec in ("fp64", "fp32"):
        F = hb.hodlr_factor(D, U, V, L, r, prec)
        sizes = [hb.hodlr_solve_workspace_size(F, k) for k in range(1, 33)]
        start = 2 if prec == "fp32" else 0  # one FP32 column also keeps its projection parts
        assert all(a <= b for a, b in zip(sizes[start:], sizes[start + 1:]))


# ------------------------------------------------------------- strong coupling
class Plain:
    """The factorization's formulas as they stand, in NumPy FP64: leaf LUs, the explicit
    inverses of K~ from the Schur complement, one right-hand side after the other
    through the levels. Its error is what FP64 roundings of these formulas cost."""

    def __init__(self, D, U, V, L, strength=None):
        self.V, self.L, self.N, self.r = V, L, U.shape[0], U.shape[1] // L
        self.D, self.U, self.inv = D, U, {}
        r = self.r
        Y = np.concatenate([np.linalg.solve(d, u) for d, u in zip(D, U.reshape(len(D), -1, U.shape[1]))])
        for c in range(L, 0, -1):
            n, q, anc = self.N >> c, slice((c - 1) * r, c * r), (c - 1) * r
            T = [V[i * n:(i + 1) * n, q].T @ Y[i * n:(i + 1) * n, q] for i in range(1 << c)]
            if strength:  # rescale the level's bases: |T| = strength in the 2-norm
                for i, t in enumerate(T):
                    f = strength / np.linalg.norm(t, 2)
                    self.U[i * n:(i + 1) * n, q] *= f
                    Y[i * n:(i + 1) * n, q] *= f
                    T[i] = t * f
            for p in range(1 << (c - 1)):
                Ta, Tb = T[2 * p], T[2 * p + 1]
                S = np.linalg.inv(np.eye(r) - Ta @ Tb)
                M = S @ Ta
                self.inv[c, p] = np.block([[np.eye(r) + Tb @ M, -Tb @ S], [-M, S]])
                a, b = slice(2 * p * n, (2 * p + 1) * n), slice((2 * p + 1) * n, (2 * p + 2) * n)
                s = np.concatenate([V[b, q].T @ Y[b, :anc], V[a, q].T @ Y[a, :anc]])
                w = self.inv[c, p] @ s
                Y[a, :anc] -= Y[a, q] @ w[:r]
                Y[b, :anc] -= Y[b, q] @ w[r:]
        self.Y = Y

    def solve(self, x, trans):
        x, r = x.copy(), self.r
        leaves = x.reshape(len(self.D), -1, x.shape[1])
        if not trans:
            x = np.concatenate([np.linalg.solve(d, b) for d, b in zip(self.D, leaves)])
        P, Q = (self.Y, self.V) if trans else (self.V, self.Y)
        for c in range(1, self.L + 1) if trans else range(self.L, 0, -1):
            n, q = self.N >> c, slice((c - 1) * r, c * r)
            for p in range(1 << (c - 1)):
                a, b = slice(2 * p * n, (2 * p + 1) * n), slice((2 * p + 1) * n, (2 * p + 2) * n)
                s = [P[a, q].T @ x[a], P[b, q].T @ x[b]]
                w = self.inv[c, p].T @ np.concatenate(s) if trans else self.inv[c, p] @ np.concatenate(s[::-1])
                first, second = (r, 0) if trans else (0, r)
                x[a] -= Q[a, q] @ w[first:first + r]
                x[b] -= Q[b, q] @ w[second:second + r]
        if trans:
            x = np.concatenate([np.linalg.solve(d.T, b) for d, b in zip(self.D, x.reshape(leaves.shape))])
        return x

    def grad(self, B):
        """(dD, dU, dV, dB) of sum b^T A^{-1} b + log|det A| through the factorization."""
        L, r, N, V, U, Y = self.L, self.r, self.N, self.V, self.U, self.Y

        def pairs(c):  # (node's rows, sibling's rows, node) of level c
            n = N >> c
            return [(slice(i * n, (i + 1) * n), slice((i ^ 1) * n, ((i ^ 1) + 1) * n), i) for i in range(1 << c)]

        X, Lam = self.solve(B, False), self.solve(B, True)
        dU, dV, Pb, Z = np.zeros_like(U), np.zeros_like(V), np.zeros_like(U), V.copy()
        cols = [slice((c - 1) * r, c * r) for c in range(L + 1)]
        for c in range(2, L + 1):
            t = {}
            for a, b, i in pairs(c):
                t[i] = Y[a, cols[c]].T @ Z[a, :r * (c - 1)]
            for a, b, i in pairs(c):
                w = self.inv[c, i >> 1].T @ np.concatenate([t[i & ~1], t[i | 1]])
                Z[a, :r * (c - 1)] -= V[a, cols[c]] @ (w[:r] if i & 1 else w[r:])
        Z = np.concatenate([np.linalg.solve(d.T, z) for d, z in zip(self.D, Z.reshape(len(self.D), -1, r * L))])
        for c in range(1, L + 1):
            for a, b, i in pairs(c):
                K = self.inv[c, i >> 1]
                H = K[r:, :r].T if i & 1 else K[:r, r:].T
                dU[a, cols[c]] += Z[a, cols[c]] @ H - Lam[a] @ (X[b].T @ V[b, cols[c]])
                dV[a, cols[c]] += Y[a, cols[c]] @ H.T - X[a] @ (Lam[b].T @ U[b, cols[c]])
                Pb[a, cols[c]] = -Z[a, cols[c]] @ H
        for c in range(2, L + 1):
            for j in range(1, c):
                for a, b, i in pairs(c):
                    dU[a, cols[c]] += Pb[a, cols[j]] @ (Y[b, cols[j]].T @ V[b, cols[c]])
                    dV[a, cols[c]] += Y[a, cols[j]] @ (Pb[b, cols[j]].T @ U[b, cols[c]])
        dD = np.stack([np.linalg.inv(self.D[i]).T - Lam[a] @ X[a].T + Pb[a] @ Y[a].T for a, b, i in pairs(L)])
        return dD, dU, dV, X + Lam


@pytest.mark.parametrize("L,r,strength", [(1, 16, 10.0), (1, 32, 1e2), (1, 48, 1e3), (1, 64, 1e4), (1, 32, 1e4),
                                          (3, 16, 1e3), (3, 32, 10.0), (3, 48, 1e2), (3, 64, 1e3), (3, 32, 1e4)])
def test_strong_coupling(cuda_lib, L, r, strength):
    """Off-diagonal blocks that dominate: |T| >> 1, where K~^{-1} and S^{-1} are small
    against the identity. Solutions, transposed solutions and gradients stay as close
    to the exact ones as the same formulas in FP64 (eight times that for the different
    order of the sums)."""
    from oracle.hodlr import assemble_dense, dense_grad
    hb = cuda_lib
    m, rng = max(64, r), np.random.default_rng(r + L)
    N = m << L
    D = rng.standard_normal((1 << L, m, m)) / np.sqrt(m) + 4 * np.eye(m)
    U, V, B = (rng.standard_normal((N, q)) for q in (r * L, r * L, 64))
    plain = Plain(D, U, V, L, strength)
    A = assemble_dense(D, U, V, L)
    Al, Bl = A.astype(np.longdouble), B.astype(np.longdouble)
    dev = [torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T for a in (U, V, B)]
    Dt = torch.from_numpy(D).cuda().transpose(1, 2).contiguous().transpose(1, 2)
    F = hb.hodlr_factor(Dt, dev[0], dev[1], L, r, "fp64")
    for trans, call in ((False, hb.hodlr_solve), (True, hb.hodlr_solve_adjoint)):
        M = A.T if trans else A
        X = np.linalg.solve(M, B).astype(np.longdouble)
        for _ in range(3):  # refined in extended precision: the exact solution to FP64's last bit
            X += np.linalg.solve(M, (Bl - (Al.T if trans else Al) @ X).astype(float))
        own = np.linalg.norm((plain.solve(B, trans) - X).astype(float)) / np.linalg.norm(X.astype(float))
        for k in (1, 4, 8, 64):
            got = call(F, dev[2][:, :k].T.clone().T).cpu().numpy()
            err = np.linalg.norm((got - X[:, :k]).astype(float)) / np.linalg.norm(X[:, :k].astype(float))
            assert err <= 8 * own, (trans, k, err, own)
    # gradients, against dense ones whose own error is cond(A) u
    k = 8
    got = hb.hodlr_grad(F, dev[0], dev[1], dev[2][:, :k].T.clone().T)[1:]
    Bk = np.ascontiguousarray(B[:, :k])
    for g, own, want in zip(got, plain.grad(Bk), dense_grad(D, U, V, L, Bk)):
        err = np.abs(g.cpu().numpy() - want).max()
        assert err <= 8 * np.abs(own - want).max() + 64 * np.linalg.cond(A) * 2.0 ** -53 * np.abs(want).max()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "tf32", "bf16"])
@pytest.mark.parametrize("m,L,r", [(1, 3, 1), (64, 6, 8), (200, 4, 64), (128, 9, 32)])
def test_solve_workspace_is_monotone(cuda_lib, m, L, r, prec):
    """The same for every precision and from one column on."""
    hb = cuda_lib
    _, (D, U, V, _) = case(m, L, r, 1, seed=1)
    F = hb.hodlr_factor(D, U, V, L, r, prec)
    sizes = [hb.hodlr_solve_workspace_size(F, k) for k in range(1, 33)]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))
