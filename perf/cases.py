"""Performance cases of the HODLR solver: what its users run, through the
binding's entry points, from single small solves to operators of 2^20 rows.

A case is a dict of plain values: ``kind`` (what is called), the tree (leaf
size ``m``, ``L`` levels, N = m 2^L), the rank ``r``, the number of columns
``k`` and, where the call takes one, the factor's precision ``prec`` or the
construction's ``kernel``. The operators are the synthetic family of
``synth.generators`` (drawn here on the GPU), except the boundary-integral one
of the headline benchmark, which the library itself constructs.
"""
import math

import torch

from paper_2208_06290_gb300 import binding as hb
from paper_2208_06290_gb300 import costs


def listed():
    return [
        # One right-hand side on a small factored operator, as inside a time step
        # or a line search: latency and launches are all there is.
        dict(name="solve-4k", kind="solve", m=64, L=6, r=16, k=1),
        # The smallest benchmark configuration: factor, solve and determinant.
        dict(name="direct-4k", kind="direct", m=64, L=6, r=16, k=1, prec="fp64"),
        # The plain FP64 direct solver at an ordinary size.
        dict(name="direct-128k", kind="direct", m=128, L=10, r=32, k=1, prec="fp64"),
        # The same on a tree that is no power of two, with an odd rank and a few columns.
        dict(name="direct-ragged", kind="direct", m=100, L=9, r=21, k=5, prec="fp64"),
        # Many right-hand sides against a stored FP64 factor, forward and transposed
        # (parameter studies, adjoint sensitivities).
        dict(name="solves-256k", kind="solves", m=256, L=10, r=32, k=64),
        # The headline: BF16 factor, FGMRES to 1e-10 and the determinant of the
        # 2^20-node boundary-integral operator.
        dict(name="gmres-bie-1m", kind="gmres", m=128, L=13, r=32, k=1, prec="bf16"),
        # Kernel-matrix shape (leaf 256, rank 64) with 16 columns: FP32 factor, refined.
        dict(name="refine-256k", kind="refine", m=256, L=10, r=64, k=16, prec="fp32"),
        # 64 columns refined with a BF16 factor on a larger tree.
        dict(name="refine-512k", kind="refine", m=256, L=11, r=32, k=64, prec="bf16"),
        # The operator applied to one vector (residuals, outer Krylov methods).
        dict(name="matvec-1m", kind="matvec", m=128, L=13, r=32, k=1),
        # The operator applied to a block of vectors (block methods, sampling).
        dict(name="matvec-256k", kind="matvec", m=256, L=10, r=64, k=32),
        # Training step of a Gaussian-process likelihood: factor and all gradients.
        dict(name="grad-16k", kind="grad", m=256, L=6, r=64, k=32, prec="fp64"),
        # Construction of a kernel operator from points.
        dict(name="compress-128k", kind="compress", m=256, L=9, r=64, k=0, kernel="matern32"),
    ]


# kind: (weight, most rows, most columns)
_RANGES = {
    "solve": (2, 1 << 17, 4),
    "solves": (2, 1 << 18, 64),
    "direct": (4, 1 << 18, 8),
    "gmres": (2, 1 << 18, 2),
    "refine": (3, 1 << 18, 64),
    "matvec": (4, 1 << 18, 64),
    "grad": (2, 1 << 14, 32),
    "compress": (1, 1 << 16, 0),
}


def draw(rng):
    kinds = list(_RANGES)
    kind = rng.choices(kinds, [_RANGES[q][0] for q in kinds])[0]
    _, most, kmost = _RANGES[kind]
    n = math.exp(rng.uniform(math.log(2048), math.log(most)))
    # a power of two, a multiple of 16 or any leaf size at all
    m = rng.choice([64, 128, 256, 16 * rng.randint(3, 16), rng.randint(33, 256)])
    L = max(1, int(math.log2(n / m)))
    r = rng.choice([8, 16, 32, 64, rng.randint(4, 64)])
    k = max(1, round(math.exp(rng.uniform(0, math.log(kmost))))) if kmost else 0
    case = dict(kind=kind, m=m, L=L, r=min(r, m), k=k)
    if kind in ("direct", "grad"):
        case["prec"] = "fp64"
    if kind in ("gmres", "refine"):
        case["prec"] = rng.choice(["fp32", "tf32", "bf16"])
    if kind == "compress":
        case["kernel"] = rng.choice(["gaussian", "matern32"])
    return case


# ------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _synthetic(case, g):
    """D = N(0, 1) / sqrt(m) + shift I, bases N(0, 1) / (2 sqrt(node size))."""
    m, L, r = case["m"], case["L"], case["r"]
    n = m << L
    d = torch.randn(1 << L, m, m, generator=g, device="cuda", dtype=torch.float64) / math.sqrt(m)
    d.diagonal(dim1=1, dim2=2).add_(8.0 if m > 128 or r > 32 else 4.0)
    u = torch.randn(r * L, n, generator=g, device="cuda", dtype=torch.float64)
    v = torch.randn(r * L, n, generator=g, device="cuda", dtype=torch.float64)
    for c in range(1, L + 1):
        u[(c - 1) * r:c * r] *= 0.5 / math.sqrt(n >> c)
        v[(c - 1) * r:c * r] *= 0.5 / math.sqrt(n >> c)
    return d.transpose(1, 2), u.T, v.T


def _columns(n, k, g):
    return torch.randn(k, n, generator=g, device="cuda", dtype=torch.float64).T


def _points(n, levels, dim, g):
    """n uniform points in the cluster tree's order (median splits, axes in turn)."""
    p = torch.rand(n, dim, generator=g, device="cuda", dtype=torch.float64)
    for c in range(levels):
        p = p.view(1 << c, n >> c, dim)
        order = p[..., c % dim].argsort(dim=1)
        p = p.gather(1, order[..., None].expand(-1, -1, dim))
    return p.reshape(n, dim).contiguous()


_KERNEL = {"gaussian": dict(dim=2, scale=0.1, nugget=1e-2), "matern32": dict(dim=3, scale=0.2, nugget=1e-3)}


def _operator(case, g):
    m, L, r = case["m"], case["L"], case["r"]
    if case["kind"] == "gmres" and case["m"] << case["L"] >= 1 << 20:
        return hb.hodlr_compress(m << L, L, r, "bie_star")
    return _synthetic(case, g)


def prepare(case, seed):
    g = _generator(seed)
    m, L, r, k = case["m"], case["L"], case["r"], case["k"]
    n = m << L
    if case["kind"] == "compress":
        return dict(case=case, points=_points(n, L, _KERNEL[case["kernel"]]["dim"], g))
    d, u, v = _operator(case, g)
    state = dict(case=case, D=d, U=u, V=v, B=_columns(n, k, g))
    if case["kind"] in ("solve", "solves"):
        state["F"] = hb.hodlr_factor(d, u, v, L, r, "fp64")
        state["X"] = torch.empty_like(state["B"])
    if case["kind"] == "matvec":
        state["Y"] = torch.empty_like(state["B"])
    return state


# --------------------------------------------------------------------- calls
def run(state):
    case = state["case"]
    kind, m, L, r = case["kind"], case["m"], case["L"], case["r"]
    if kind == "compress":
        q = _KERNEL[case["kernel"]]
        return list(hb.hodlr_compress(m << L, L, r, case["kernel"], state["points"], scale=q["scale"],
                                      nugget=q["nugget"]))
    D, U, V, B = state["D"], state["U"], state["V"], state["B"]
    if kind == "matvec":
        return [hb.hodlr_matvec(D, U, V, L, r, B, state["Y"])]
    if kind == "solve":
        return [hb.hodlr_solve(state["F"], state["X"].copy_(B))]
    if kind == "solves":
        return [hb.hodlr_solve(state["F"], state["X"].copy_(B)), hb.hodlr_solve_adjoint(state["F"], B.clone())]
    F = hb.hodlr_factor(D, U, V, L, r, case["prec"])
    if kind == "direct":
        x = hb.hodlr_solve(F, B.clone())
    elif kind == "gmres":
        x = hb.hodlr_gmres(F, D, U, V, B, tol=1e-10)[0]
    elif kind == "refine":
        return [hb.hodlr_solve_refined(F, D, U, V, B, tol=1e-10)[0]]
    else:
        loss, dD, dU, dV, dB = hb.hodlr_grad(F, U, V, B)
        return [loss, dD, dU, dV, dB]
    sign, logabsdet = hb.hodlr_logdet(F)
    return [x, sign, logabsdet]


def work(case):
    kind, m, L, r, k = case["kind"], case["m"], case["L"], case["r"], case["k"]
    n = m << L
    operator = 8.0 * costs.storage_elems(n, m, r, L)
    columns = 16.0 * n * k
    solve = costs.solve_flops(n, m, r, L, k)
    if kind == "compress":
        return dict(bytes=operator, flops=2.0 * n * r * r * L)
    if kind == "matvec":
        return dict(bytes=operator + columns, flops=costs.matvec_flops(n, m, r, L, k))
    if kind in ("solve", "solves"):
        passes = 2 if kind == "solves" else 1
        factor = operator + 8.0 * 4 * r * r * ((1 << L) - 1)
        return dict(bytes=passes * (factor + columns), flops=passes * solve)
    factor = costs.factor_flops(n, m, r, L)
    if kind == "direct":
        return dict(bytes=operator + columns, flops=factor + solve)
    if kind in ("gmres", "refine"):
        return dict(bytes=operator + columns, flops=factor + solve + costs.matvec_flops(n, m, r, L, k))
    gradient = (2.0 * solve + 2.0 * n * m * k + 8.0 * n * r * L * k  # both solves, the terms of the columns
                + 2.0 * n * r * r * L * L + 2.0 * m * n * r * L      # the adjoint bases
                + 4.0 * n * r * r * L * (L - 1)                      # each node's term on what lies below it
                + 2.0 * m * m * n + 2.0 * m * n * r * L)             # the leaves
    return dict(bytes=2.0 * (operator + columns), flops=factor + gradient)


# ------------------------------------------------------------- 64-bit values
def _solve64(D, U, V, L, r, B):
    """A^{-1} B and log|det A|: the level-by-level elimination with torch's own
    LU and products."""
    n, k = B.shape
    c_top = r * L
    lu, piv, _ = torch.linalg.lu_factor_ex(D.contiguous())
    z = torch.cat([U, B], dim=1).view(1 << L, n >> L, c_top + k)
    z = torch.linalg.lu_solve(lu, piv, z.contiguous()).reshape(n, c_top + k)
    logdet = lu.diagonal(dim1=1, dim2=2).abs().log().sum()
    del lu
    for c in range(L, 0, -1):
        nodes, rows = 1 << c, n >> c
        own = z[:, (c - 1) * r:c * r].reshape(nodes, rows, r)
        rest = torch.cat([z[:, :(c - 1) * r], z[:, c_top:]], dim=1).view(nodes, rows, -1)
        vt = V[:, (c - 1) * r:c * r].reshape(nodes, rows, r).transpose(1, 2)
        t = (vt @ own).view(nodes // 2, 2, r, r)
        s = (vt @ rest).view(nodes // 2, 2, r, -1)
        eye = torch.eye(r, device=B.device, dtype=B.dtype).expand(nodes // 2, r, r)
        kk = torch.cat([torch.cat([eye, t[:, 1]], 2), torch.cat([t[:, 0], eye], 2)], 1)
        w = torch.linalg.solve(kk, torch.cat([s[:, 1], s[:, 0]], 1)).reshape(nodes, r, -1)
        logdet = logdet + torch.linalg.slogdet(kk)[1].sum()
        rest = torch.baddbmm(rest, own, w, alpha=-1.0).view(n, -1)
        z[:, :(c - 1) * r] = rest[:, :(c - 1) * r]
        z[:, c_top:] = rest[:, (c - 1) * r:]
    return z[:, c_top:].T.contiguous().T, float(logdet)


def _matvec64(D, U, V, L, r, X):
    n, k = X.shape
    y = (D @ X.reshape(1 << L, n >> L, k)).reshape(n, k)
    for c in range(1, L + 1):
        nodes, rows = 1 << c, n >> c
        u = U[:, (c - 1) * r:c * r].reshape(nodes, rows, r)
        v = V[:, (c - 1) * r:c * r].reshape(nodes, rows, r)
        s = v.transpose(1, 2) @ X.reshape(nodes, rows, k)
        s = s.view(nodes // 2, 2, r, k).flip(1).reshape(nodes, r, k)
        y += (u @ s).view(n, k)
    return y.T.contiguous().T


def _dense(D, U, V, L, r):
    n, m = U.shape[0], U.shape[0] >> L
    a = torch.zeros(n, n, device="cuda", dtype=torch.float64)
    for b in range(1 << L):
        a[b * m:(b + 1) * m, b * m:(b + 1) * m] = D[b]
    for c in range(1, L + 1):
        rows = n >> c
        for i in range(1 << c):
            j, q = i ^ 1, slice((c - 1) * r, c * r)
            a[i * rows:(i + 1) * rows, j * rows:(j + 1) * rows] = \
                U[i * rows:(i + 1) * rows, q] @ V[j * rows:(j + 1) * rows, q].T
    return a


def _grad64(D, U, V, L, r, B):
    n, m = U.shape[0], U.shape[0] >> L
    inv = torch.linalg.inv(_dense(D, U, V, L, r))
    X, Lam = inv @ B, inv.T @ B
    loss = float((B * X).sum()) + _solve64(D, U, V, L, r, B[:, :1])[1]
    G = inv.T - Lam @ X.T
    dD = torch.stack([G[b * m:(b + 1) * m, b * m:(b + 1) * m] for b in range(1 << L)])
    dU, dV = torch.empty_like(U), torch.empty_like(V)
    for c in range(1, L + 1):
        rows, q = n >> c, slice((c - 1) * r, c * r)
        for i in range(1 << c):
            a, b = slice(i * rows, (i + 1) * rows), slice((i ^ 1) * rows, ((i ^ 1) + 1) * rows)
            dU[a, q] = G[a, b] @ V[b, q]
            dV[b, q] = G[a, b].T @ U[a, q]
    return [loss, dD, dU, dV, X + Lam]


def exact(case, seed):
    kind, m, L, r = case["kind"], case["m"], case["L"], case["r"]
    n = m << L
    g = _generator(seed)
    if kind == "compress":  # the leaf blocks; the bases follow from the cross approximation's own pivots
        q = _KERNEL[case["kernel"]]
        p = _points(n, L, q["dim"], g).view(1 << L, m, q["dim"])
        dist = (p[:, :, None, :] - p[:, None, :, :]).square().sum(-1).sqrt()
        if case["kernel"] == "gaussian":
            blocks = torch.exp(-dist.square() / (2 * q["scale"] ** 2))
        else:
            t = math.sqrt(3.0) * dist / q["scale"]
            blocks = (1 + t) * torch.exp(-t)
        blocks.diagonal(dim1=1, dim2=2).add_(q["nugget"])
        return [blocks, None, None]
    D, U, V = _operator(case, g)
    B = _columns(n, case["k"], g)
    if kind == "matvec":
        return [_matvec64(D, U, V, L, r, B)]
    if kind == "grad":
        return _grad64(D, U, V, L, r, B) if n <= 1 << 14 else None
    x, logdet = _solve64(D, U, V, L, r, B)
    if kind == "solve" or kind == "refine":
        return [x]
    if kind == "solves":
        return [x, _solve64(D.transpose(1, 2), V, U, L, r, B)[0]]
    return [x, None, logdet]
