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
