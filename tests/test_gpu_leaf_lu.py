"""Leaf LU with partial pivoting: panel edges, rows that have to move, ties, zero
and non-finite blocks (GPU).

Leaves here are plain N(0, 1) blocks or blocks of small whole numbers, so almost
every column exchanges rows. Solves are checked by their normwise backward error
|b - A x| / (|A| |x| + |b|), which Gaussian elimination with partial pivoting
keeps below n^2 u times its growth factor (taken as n^(2/3), the average of
random matrices, times four).
"""
import numpy as np
import pytest
import torch

from oracle.hodlr import assemble_dense
from synth import HodlrShape, gaussian_rhs, synthetic_hodlr, to_math

pytestmark = pytest.mark.gpu


def case(m, L, r, k, seed, whole=False):
    N = m << L
    D, U, V, g = synthetic_hodlr(HodlrShape(N, L, r), 0.0, seed)
    rng = np.random.default_rng(seed)
    blocks = rng.integers(-2, 3, (1 << L, m, m)).astype(float) if whole else rng.standard_normal((1 << L, m, m))
    if whole:  # unit triangular factors with their rows shuffled: invertible, full of ties
        lo = np.tril(rng.integers(-1, 2, (1 << L, m, m)), -1) * (np.arange(m)[:, None] - np.arange(m) <= 3)
        up = np.triu(rng.integers(-1, 2, (1 << L, m, m)), 1) * (np.arange(m) - np.arange(m)[:, None] <= 3)
        blocks = (lo + np.eye(m)) @ (up + np.eye(m))
        blocks = np.stack([b[rng.permutation(m)] for b in blocks]).astype(float)
    D = torch.from_numpy(blocks).transpose(1, 2).contiguous().transpose(1, 2)
    B = gaussian_rhs(N, k, g)
    return to_math(D, U, V, B), tuple(t.to("cuda") for t in (D, U, V, B))


def backward_error(Dm, Um, Vm, L, x, b):
    A = assemble_dense(Dm, Um, Vm, L)
    return np.linalg.norm(b - A @ x) / (np.linalg.norm(A) * np.linalg.norm(x) + np.linalg.norm(b)), A


@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 63, 64, 65, 96, 100, 127, 128, 129, 160, 225, 255, 256])
def test_leaf_lu_fp64(cuda_lib, m):
    hb = cuda_lib
    L, r, k = 2, min(4, m), 6
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=m)
    F = hb.hodlr_factor(D, U, V, L, r, "fp64")
    n = m << L
    for cols in (1, k):
        x = hb.hodlr_solve(F, B[:, :cols].T.clone().T).cpu().numpy()
        err, A = backward_error(Dm, Um, Vm, L, x, Bm[:, :cols])
        assert err <= 4 * n ** (2 + 2 / 3) * 2.0 ** -53
    s, la = hb.hodlr_logdet(F)
    so, lao = np.linalg.slogdet(A)
    assert s == so
    # each of the n pivots carries a relative error of at most cond(A) u n
    assert abs(la - lao) <= n * n * np.linalg.cond(A) * 2.0 ** -53


@pytest.mark.parametrize("m", [129, 160, 191, 224, 250, 256])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_leaf_lu_fp32(cuda_lib, m, prec):
    """Leaves above 128 rows are FP32 LUs in the low-precision factors; with zero
    bases the factor is its leaves, whatever the panels' precision."""
    hb = cuda_lib
    L, r, k = 2, 4, 3
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=m + 1)
    U.zero_()
    F = hb.hodlr_factor(D, U, V, L, r, prec)
    for b in range(1 << L):
        q = slice(b * m, (b + 1) * m)
        x = hb.hodlr_solve(F, B.clone()).cpu().numpy()[q]
        res = np.linalg.norm(Bm[q] - Dm[b] @ x) / (np.linalg.norm(Dm[b]) * np.linalg.norm(x) + np.linalg.norm(Bm[q]))
        assert res <= 4 * m ** (2 + 2 / 3) * 2.0 ** -24 / np.sqrt(m)  # roundings add up as a random walk
    s, la = hb.hodlr_logdet(F)
    ref = [np.linalg.slogdet(Dm[b]) for b in range(1 << L)]
    assert s == np.prod([q[0] for q in ref])
    cond = max(np.linalg.cond(Dm[b]) for b in range(1 << L))
    assert abs(la - sum(q[1] for q in ref)) <= len(ref) * m * cond * 2.0 ** -24


@pytest.mark.parametrize("m", [40, 100, 256])
def test_leaf_lu_ties(cuda_lib, m):
    """Determinant +-1 blocks of whole numbers: every pivot column has ties."""
    hb = cuda_lib
    L, r, k = 2, 4, 2
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=m + 2, whole=True)
    U.zero_()
    F = hb.hodlr_factor(D, U, V, L, r, "fp64")
    s, la = hb.hodlr_logdet(F)
    assert s == np.prod([np.linalg.slogdet(b)[0] for b in Dm])
    assert abs(la) <= len(Dm) * m * m * 2.0 ** -53 * max(np.linalg.cond(b) for b in Dm)


@pytest.mark.parametrize("m,prec", [(48, "fp64"), (200, "fp64"), (200, "fp32")])
@pytest.mark.parametrize("row", [0, 30, 45])
def test_leaf_lu_bad_blocks(cuda_lib, m, prec, row):
    hb = cuda_lib
    L, r = 2, 4
    _, (D, U, V, B) = case(m, L, r, 1, seed=3)
    Dz = D.clone().transpose(1, 2).contiguous().transpose(1, 2)
    Dz[2, :, row] = 0.0  # a zero column is a zero pivot there
    with pytest.raises(hb.HodlrError) as e:
        hb.hodlr_logdet(hb.hodlr_factor(Dz, U, V, L, r, prec))
    assert (e.value.code, e.value.where, e.value.detail) == (hb.HODLR_ERR_SINGULAR_LEAF, 2, row)
    Dn = D.clone().transpose(1, 2).contiguous().transpose(1, 2)
    Dn[1, row, m - 1] = float("nan")
    with pytest.raises(hb.HodlrError) as e:
        hb.hodlr_logdet(hb.hodlr_factor(Dn, U, V, L, r, prec))
    assert e.value.code == hb.HODLR_ERR_NONFINITE


def smooth_block(rng, m, nugget):
    x = rng.random((m, 2)) * 0.25
    d2 = ((x[:, None] - x[None]) ** 2).sum(-1)
    return np.exp(-d2 / 0.02) + nugget * np.eye(m)


@pytest.mark.parametrize("m", [20, 64, 100, 256])
@pytest.mark.parametrize("nugget", [1e-2, 1e-6, 1e-8, 1e-10])
def test_ill_conditioned_leaves(cuda_lib, m, nugget):
    """Leaves of a smooth kernel, condition numbers 1e3 to 1e12, whose pivots fall by
    as much within one block: solves stay as backward stable as substitution with
    LAPACK's factors (eight times its error for other orders of the sums, and never
    held below one rounding)."""
    import scipy.linalg
    hb = cuda_lib
    L, r, k = 2, 4, 64
    rng = np.random.default_rng(m)
    Dm = np.stack([smooth_block(rng, m, nugget) for _ in range(1 << L)])
    Bm = rng.standard_normal((m << L, k))
    D = torch.from_numpy(Dm).cuda().transpose(1, 2).contiguous().transpose(1, 2)
    B = torch.from_numpy(np.ascontiguousarray(Bm.T)).cuda().T
    Z = torch.zeros(r * L, m << L, dtype=torch.float64, device="cuda").T
    F = hb.hodlr_factor(D, Z, Z, L, r, "fp64")

    def backward(A, x, b):
        res = np.linalg.norm((b - A.astype(np.longdouble) @ x).astype(float), axis=0)
        return (res / (np.linalg.norm(A) * np.linalg.norm(x, axis=0) + np.linalg.norm(b, axis=0))).max()

    for trans, call in ((0, hb.hodlr_solve), (1, hb.hodlr_solve_adjoint)):
        for cols in (1, 3, 8, k):
            x = call(F, B[:, :cols].T.clone().T).cpu().numpy()
            for i, d in enumerate(Dm):
                q, A = slice(i * m, (i + 1) * m), d.T if trans else d
                own = scipy.linalg.lu_solve(scipy.linalg.lu_factor(d), Bm[q, :cols], trans=trans)
                err, ref = backward(A, x[q], Bm[q, :cols]), backward(A, own, Bm[q, :cols])
                assert err <= max(8 * ref, 2.0 ** -53), (trans, cols, i, err, ref)


@pytest.mark.parametrize("m", [1, 31, 32, 33, 65, 100, 128, 129, 256])
def test_leaf_lu_matches_cpu_lu(cuda_lib, m):
    """Plain normal blocks, rows exchanged in almost every column: backward errors and
    determinants within a small factor of an FP64 LU on the CPU."""
    import scipy.linalg
    hb = cuda_lib
    L, r, k = 2, 1, 6
    (Dm, Um, Vm, Bm), (D, U, V, B) = case(m, L, r, k, seed=m + 5)
    U.zero_()
    F = hb.hodlr_factor(D, U, V, L, r, "fp64")
    lus = [scipy.linalg.lu_factor(d) for d in Dm]
    for cols in (1, k):
        x = hb.hodlr_solve(F, B[:, :cols].T.clone().T).cpu().numpy()
        for i, d in enumerate(Dm):
            q = slice(i * m, (i + 1) * m)
            err = [np.linalg.norm(Bm[q, :cols] - d @ y) / (np.linalg.norm(d) * np.linalg.norm(y))
                   for y in (x[q], scipy.linalg.lu_solve(lus[i], Bm[q, :cols]))]
            assert err[0] <= max(8 * err[1], 2 * 2.0 ** -53), (cols, i, err)
    s, la = hb.hodlr_logdet(F)
    diag = np.concatenate([np.diag(f[0]) for f in lus])
    ref = np.log(np.abs(diag)).sum()
    # the product of the pivots is the determinant of blocks A + E with |E| as bounded above
    pert = sum(8 * np.sqrt(m) * 2.0 ** -53 * np.linalg.norm(np.linalg.inv(d)) * np.linalg.norm(d) for d in Dm)
    assert abs(la - ref) <= pert + len(diag) * 2.0 ** -53 * np.abs(np.log(np.abs(diag))).max()
    assert s == np.prod([np.linalg.slogdet(d)[0] for d in Dm])
