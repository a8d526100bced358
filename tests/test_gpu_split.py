"""FP64 products formed on the FP16 tensor cores from split operands: the edges
of their tiles and digits (GPU).

The matvec bound is element-wise and rigorous: two FP64 evaluations of
y = A x that round every product and sum differ by at most
2 (m + sum_c (n_c + r) + L + 1) u (|A| |x|)_i with |A| |x| formed from the
blocks' absolute values, u = 2^-53.
"""
import numpy as np
import pytest
import torch

from oracle.hodlr import RecursiveHODLR, matvec as o_matvec
from synth import HodlrShape, gaussian_rhs, synthetic_hodlr, to_math

pytestmark = pytest.mark.gpu
U64 = 2.0 ** -53


def case(m, L, r, k, seed):
    N = m << L
    D, U, V, g = synthetic_hodlr(HodlrShape(N, L, r), 4.0, seed)
    B = gaussian_rhs(N, k, g)
    return to_math(D, U, V, B), tuple(t.to("cuda") for t in (D, U, V, B))


def matvec_bound(D, U, V, L, X):
    N, r = U.shape[0], U.shape[1] // L
    terms = (N >> L) + sum((N >> c) + r for c in range(1, L + 1)) + L + 1
    return 2 * terms * U64 * o_matvec(np.abs(D), np.abs(U), np.abs(V), L, np.abs(X))


# row tiles of 16 / 64 / 128, 32-row blocks, 8 / 16 / 32 / 64-column tiles, rank
# tiles of 16 and 32, chunks that are no multiple of 64 or 4 rows
@pytest.mark.parametrize("m,L,r,k", [
    (1, 2, 1, 2), (15, 2, 3, 3), (16, 1, 16, 8), (17, 3, 17, 9), (31, 2, 15, 16), (33, 5, 31, 17), (64, 4, 32, 32),
    (100, 4, 33, 33), (127, 1, 64, 64), (129, 2, 48, 65), (250, 3, 63, 5), (256, 3, 64, 2), (65, 5, 8, 7)])
def test_split_matvec_edges(cuda_lib, m, L, r, k):
    (Dm, Um, Vm, Xm), (D, U, V, X) = case(m, L, r, k, seed=m + 7 * r + k)
    Y = cuda_lib.hodlr_matvec(D, U, V, L, r, X).cpu().numpy()
    assert (np.abs(Y - o_matvec(Dm, Um, Vm, L, Xm)) <= matvec_bound(Dm, Um, Vm, L, Xm)).all()


@pytest.mark.parametrize("scale", [1e-300, 2.0 ** -401, 2.0 ** -399, 2.0 ** 399, 2.0 ** 402, 1e250])
def test_split_matvec_range(cuda_lib, scale):
    """Vectors inside and outside the exponents that the digits cover, beside an
    all-zero column and one with a spread of 30 orders of magnitude."""
    m, L, r, k = 64, 3, 16, 9
    (Dm, Um, Vm, Xm), (D, U, V, _) = case(m, L, r, k, seed=5)
    Xm = Xm * scale
    Xm[:, 3] = 0.0
    Xm[:, 4] *= 10.0 ** np.linspace(-15, 15, Xm.shape[0])
    X = torch.from_numpy(np.ascontiguousarray(Xm.T)).cuda().T
    Y = cuda_lib.hodlr_matvec(D, U, V, L, r, X).cpu().numpy()
    # below the normal range products round to multiples of 2^-1074
    tiny = Um.shape[0] * 2.0 ** -1074
    assert (np.abs(Y - o_matvec(Dm, Um, Vm, L, Xm)) <= matvec_bound(Dm, Um, Vm, L, Xm) + tiny).all()
    assert (Y[:, 3] == 0.0).all()


def test_split_matvec_nonfinite(cuda_lib):
    """An infinity and a NaN reach the entries that FP64 arithmetic gives them to."""
    m, L, r, k = 48, 3, 5, 4
    (Dm, Um, Vm, Xm), (D, U, V, _) = case(m, L, r, k, seed=6)
    Xm[70, 1] = np.inf
    Xm[200, 2] = np.nan
    X = torch.from_numpy(np.ascontiguousarray(Xm.T)).cuda().T
    Y = cuda_lib.hodlr_matvec(D, U, V, L, r, X).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = o_matvec(Dm, Um, Vm, L, Xm)
    assert np.array_equal(np.isnan(Y), np.isnan(ref)) and np.array_equal(np.isinf(Y), np.isinf(ref))
    fine = np.isfinite(ref).all(axis=0)
    assert fine.tolist() == [True, False, False, True]
    assert (np.abs(Y - ref)[:, fine] <= matvec_bound(Dm, Um, Vm, L, Xm[:, fine].copy() if fine.all() else
                                                     np.where(np.isfinite(Xm), Xm, 0.0))[:, fine]).all()


# solutions of these operators (leaf shift 4, condition numbers of a few tens)
# agree with the oracle's to a few hundred roundings
@pytest.mark.parametrize("m,L,r,k", [(31, 3, 9, 5), (32, 2, 32, 8), (33, 4, 33, 9), (96, 3, 17, 33), (128, 3, 64, 64),
                                     (129, 2, 16, 65), (255, 2, 40, 12), (256, 2, 64, 31)])
def test_split_factor_solves(cuda_lib, m, L, r, k):
    hb = cuda_lib
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=3 * m + r)
    rec = RecursiveHODLR(Dm, Um, Vm, L)
    F = hb.hodlr_factor(D, U, V, L, r, "fp64")
    for got, ref in ((hb.hodlr_solve(F, B.clone()), rec.solve(Bm)),
                     (hb.hodlr_solve_adjoint(F, B.clone()), rec.solve_adjoint(Bm))):
        np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
    s, la = hb.hodlr_logdet(F)
    so, lao = rec.slogdet()
    assert s == so and abs(la - lao) <= 1e-12 * abs(lao)


def test_split_matvec_graded(cuda_lib):
    """Columns of A and entries of x scaled against each other by up to 2^60, as
    unknowns in unlike units are: every element of A x keeps the relative
    accuracy of its own sum |A| |x|, as with FP64 products."""
    m, L, r, k = 80, 3, 20, 12
    (Dm, Um, Vm, Xm), _ = case(m, L, r, k, seed=9)
    N = m << L
    s = 2.0 ** np.random.default_rng(9).integers(-30, 31, N)
    Dm, Vm, Xm = Dm * s.reshape(1 << L, 1, m), Vm * s[:, None], Xm / s[:, None]
    D = torch.from_numpy(np.ascontiguousarray(Dm.transpose(0, 2, 1))).cuda().transpose(1, 2)
    U, V, X = (torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T for a in (Um, Vm, Xm))
    Y = cuda_lib.hodlr_matvec(D, U, V, L, r, X).cpu().numpy()
    # digits: 2^-45 of the sum of magnitudes of every 32 or 64 terms
    bound = matvec_bound(Dm, Um, Vm, L, Xm) + 2.0 ** -44 * o_matvec(np.abs(Dm), np.abs(Um), np.abs(Vm), L, np.abs(Xm))
    assert (np.abs(Y - o_matvec(Dm, Um, Vm, L, Xm)) <= bound).all()


@pytest.mark.parametrize("m,L,r,k", [(16, 4, 3, 9), (40, 4, 16, 17), (33, 5, 17, 33), (64, 5, 32, 12), (48, 3, 33, 9),
                                     (64, 4, 47, 40), (64, 4, 64, 16)])
def test_split_coupling_and_gradient(cuda_lib, m, L, r, k):
    """Coupling systems of 2r = 6 .. 128 unknowns with 9 and more right-hand sides,
    forward and transposed, and the gradient's leaf blocks, against the oracle."""
    from oracle.hodlr import dense_grad
    hb = cuda_lib
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=m + r)
    F = hb.hodlr_factor(D, U, V, L, r, "fp64")
    rec = RecursiveHODLR(Dm, Um, Vm, L)
    for got, ref in ((hb.hodlr_solve(F, B.clone()), rec.solve(Bm)),
                     (hb.hodlr_solve_adjoint(F, B.clone()), rec.solve_adjoint(Bm))):
        np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
    loss, dD, dU, dV, dB = hb.hodlr_grad(F, U, V, B)
    ref = dense_grad(Dm, Um, Vm, L, Bm)
    for got, want in zip((dD, dU, dV, dB), ref):
        np.testing.assert_allclose(got.cpu().numpy(), want, rtol=0, atol=1e-10 * np.abs(want).max())


def fma_sums(A, X):
    """A @ X as chains of FP64 FMAs, and the exact sums, both per element."""
    exact = A.astype(np.longdouble) @ X.astype(np.longdouble)
    acc = np.zeros((A.shape[0], X.shape[1]))
    for t in range(A.shape[1]):
        acc = (acc + np.outer(A[:, t].astype(np.longdouble), X[t].astype(np.longdouble))).astype(float)
    return acc, exact


def graded(rng, shape, axis, bits):
    """Normal entries scaled by 2^-bits beside one entry of 1.5 per vector."""
    a = rng.standard_normal(shape) * 2.0 ** -bits
    at = rng.integers(0, shape[axis], shape[1 - axis])
    idx = (np.arange(len(at)), at) if axis == 1 else (at, np.arange(len(at)))
    a[idx] = 1.5
    return a


def operators_of(A, rng):
    """Matrices whose products with X are A X alone: A as leaf blocks, and A as the
    bases' products with unit vectors on either side (projections, updates)."""
    n = A.shape[0]
    zero = np.zeros((2 * n, n))
    eye = np.eye(n)
    yield "leaf", np.stack([A, A]), zero, zero
    yield "project", np.zeros((2, n, n)), np.concatenate([eye, eye]), np.concatenate([A.T, A.T])
    yield "update", np.zeros((2, n, n)), np.concatenate([A, A]), np.concatenate([eye, eye])


@pytest.mark.parametrize("n,k", [(32, 16), (64, 16), (64, 64), (32, 5)])
@pytest.mark.parametrize("bits", [0, 2, 3, 4, 5, 6, 7, 8, 12])
def test_split_small_sums(cuda_lib, n, k, bits):
    """Sums that are small beside the product of their vectors' largest entries keep
    the accuracy of FP64 FMAs: each within their bound n u Sum |a| |b|, and all
    together no further from the exact ones."""
    rng = np.random.default_rng(100 * n + k + bits)
    A, X = graded(rng, (n, n), 1, bits), graded(rng, (n, k), 0, bits)
    fma, exact = fma_sums(A, X)
    s = np.abs(A) @ np.abs(X)
    ref = np.sqrt(np.mean(((fma - exact) / s).astype(float) ** 2))
    for name, D, U, V in operators_of(A, rng):
        Xs = np.concatenate([X, X])  # the sibling's rows are the same
        Dt = torch.from_numpy(D).cuda().transpose(1, 2).contiguous().transpose(1, 2)
        Ut, Vt, Xt = (torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T for a in (U, V, Xs))
        y = cuda_lib.hodlr_matvec(Dt, Ut, Vt, 1, n, Xt).cpu().numpy()
        for half in (y[:n], y[n:]):
            err = ((half - exact) / s).astype(float)
            assert np.abs(err).max() <= n * U64, (name, np.abs(err).max() / U64)
            # 16 standard errors of a mean square of n k values
            assert np.sqrt(np.mean(err ** 2)) <= ref * (1 + 8 * np.sqrt(2.0 / (n * k))), (name, ref / U64)


@pytest.mark.parametrize("n", [32, 64])
@pytest.mark.parametrize("digits", [(0, 70, -128), (0, 127, 127), (1, 127, 127)])
def test_split_worst_digits(cuda_lib, n, digits):
    """Entries whose left-out digit products all have one sign, beside two largest
    entries that meet zeros."""
    d = list(digits[:2]) + [digits[2]] * 6
    x = sum(q * 256.0 ** (7 - i) for i, q in enumerate(d[:7])) * 2.0 ** -61  # 53 bits
    A, X = np.full((n, n), x), np.full((n, 8), x)
    A[:, 0], A[:, 1] = 1.0, 0.0
    X[0], X[1] = 0.0, 1.0
    _, exact = fma_sums(A, X)
    s = np.abs(A) @ np.abs(X)
    for name, D, U, V in operators_of(A, None):
        Dt = torch.from_numpy(D).cuda().transpose(1, 2).contiguous().transpose(1, 2)
        Ut, Vt, Xt = (torch.from_numpy(np.ascontiguousarray(a.T)).cuda().T for a in (U, V, np.concatenate([X, X])))
        y = cuda_lib.hodlr_matvec(Dt, Ut, Vt, 1, n, Xt).cpu().numpy()[:n]
        err = np.abs(((y - exact) / s).astype(float)).max()
        assert err <= n * U64, (name, err / U64)
