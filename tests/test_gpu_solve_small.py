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
