"""FP32 level stage and FP32 leaf solves of more than eight columns: the edges of
their tiles (GPU).

The operators have condition numbers of a few tens; an FP32 factor's solution is
off by a few hundred FP32 roundings at most, one with BF16 panels by a few BF16
ones (the low-rank terms are a fraction of the leaves)."""
import numpy as np
import pytest
import torch

from oracle.hodlr import RecursiveHODLR
from synth import HodlrShape, gaussian_rhs, synthetic_hodlr, to_math

pytestmark = pytest.mark.gpu
TOL = {"fp32": 300 * 2.0 ** -24, "tf32": 8 * 2.0 ** -11, "bf16": 8 * 2.0 ** -9}


# rank tiles of 32, column tiles of 64 / 128 / 256, row blocks of 8 and 16, row tiles
# of 64 and 128, row counts that are no multiple of four, leaves above and below 128
@pytest.mark.parametrize("m,L,r,k", [
    (33, 4, 9, 9), (64, 5, 32, 64), (50, 4, 33, 65), (100, 4, 48, 17), (128, 3, 64, 129), (129, 3, 31, 64),
    (130, 2, 64, 12), (161, 3, 40, 66), (191, 2, 16, 200), (250, 3, 64, 9), (256, 3, 32, 63), (256, 2, 64, 130)])
@pytest.mark.parametrize("prec", ["fp32", "tf32", "bf16"])
def test_low_precision_solves(cuda_lib, m, L, r, k, prec):
    hb = cuda_lib
    N = m << L
    D, U, V, g = synthetic_hodlr(HodlrShape(N, L, r), 4.0, m + r + k)
    B = gaussian_rhs(N, k, g)
    Dm, Um, Vm, Bm = to_math(D, U, V, B)
    rec = RecursiveHODLR(Dm, Um, Vm, L)
    D, U, V, B = (t.to("cuda") for t in (D, U, V, B))
    F = hb.hodlr_factor(D, U, V, L, r, prec)
    for got, ref in ((hb.hodlr_solve(F, B.clone()), rec.solve(Bm)),
                     (hb.hodlr_solve_adjoint(F, B.clone()), rec.solve_adjoint(Bm))):
        got = got.cpu().numpy()
        assert np.linalg.norm(got - ref) <= TOL[prec] * np.linalg.norm(ref)
        assert np.abs(got - ref).max() <= 8 * TOL[prec] * np.abs(ref).max()


def test_low_precision_solve_strided(cuda_lib):
    """Columns in a buffer with an odd leading dimension and an odd first row."""
    hb = cuda_lib
    m, L, r, k = 200, 2, 20, 70
    N = m << L
    D, U, V, g = synthetic_hodlr(HodlrShape(N, L, r), 4.0, 1)
    B = gaussian_rhs(N, k, g)
    Dm, Um, Vm, Bm = to_math(D, U, V, B)
    buf = torch.zeros(k, N + 7, dtype=torch.float64, device="cuda").T
    X = buf[3:3 + N]
    X.copy_(B)
    D, U, V = (t.to("cuda") for t in (D, U, V))
    hb.hodlr_solve(hb.hodlr_factor(D, U, V, L, r, "fp32"), X)
    ref = RecursiveHODLR(Dm, Um, Vm, L).solve(Bm)
    assert np.linalg.norm(X.cpu().numpy() - ref) <= TOL["fp32"] * np.linalg.norm(ref)
    assert (buf[:3] == 0).all() and (buf[3 + N:] == 0).all()


@pytest.mark.parametrize("m,L", [(64, 5), (80, 5), (96, 6), (112, 6), (208, 5), (128, 8)])
@pytest.mark.parametrize("prec", ["bf16", "tf32"])
def test_projections_stay_on_tensor_cores(cuda_lib, m, L, prec):
    """Every level of a BF16 or TF32 factor whose nodes, halved to at most 1024 rows, are
    whole 64-row tiles projects with the tcgen05 kernel, on small trees too."""
    hb = cuda_lib
    r, N = 32, m << L
    D, U, V, g = synthetic_hodlr(HodlrShape(N, L, r), 4.0, m)
    B = gaussian_rhs(N, 3, g)
    D, U, V, B = (t.to("cuda") for t in (D, U, V, B))
    want = 0
    for c in range(1, L + 1):
        n = N >> c
        while n > 1024:
            n //= 2
        want += n % 64 == 0
    hb.hodlr_profile_reset()
    hb.hodlr_profile_enable(True)
    try:
        F = hb.hodlr_factor(D, U, V, L, r, prec)
        got = hb.hodlr_profile_read()["project_tc"][1]
    finally:
        hb.hodlr_profile_enable(False)
        hb.hodlr_profile_reset()
    assert got == want
    X, _, rr, _ = hb.hodlr_solve_refined(F, D, U, V, B, tol=1e-10)
    assert rr <= 1e-10
    res = hb.hodlr_matvec(D, U, V, L, r, X) - B
    assert float((res.norm(dim=0) / B.norm(dim=0)).max()) <= 2e-10
