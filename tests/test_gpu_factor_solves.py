"""k = G^{-1} g from kept factors in ill-conditioned stages (GPU): as small a residual as two substitutions leave.

A product with a stored inverse of the factor leaves one that grows with the factor's condition, which the
refinement then has to make up for: more corrections, and FP32 interior-point loops that do not converge.
"""
import numpy as np
import pytest
from scipy.linalg import solve_triangular

from paper_1510_03110_gb300 import mhe, synth

from gpu_util import device_inputs

pytestmark = pytest.mark.gpu


def _stiff(rng, n, scale, dt):
    """G = I + scale V V^T with V of half the rank, and g in the range of V: a master stage's form."""
    V = rng.standard_normal((n, max(1, n // 2)))
    G = (np.eye(n) + scale * V @ V.T).astype(dt)
    G = np.tril(G) + np.tril(G, -1).T
    return G.astype(np.float64), (scale * (V @ rng.standard_normal(V.shape[1]))).astype(dt).astype(np.float64)


def _residual(G, k, g):
    """Largest entry of |G k - g| / (|G| |k| + |g|)."""
    G, k, g = (t.astype(np.longdouble) for t in (G, k, g))
    return float((np.abs(G @ k - g) / (np.abs(G) @ np.abs(k) + np.abs(g))).max())


@pytest.mark.parametrize("batch", [40, 180])   # one launch per solve (nx <= 24), one per level pass
@pytest.mark.parametrize("prec", [mhe.MHE_FP64, mhe.MHE_FP32_IR])
@pytest.mark.parametrize("n,m", [(6, 3), (12, 6), (20, 10), (20, 20), (24, 12), (64, 32)])
def test_stored_factor_solves_leave_a_small_residual(n, m, prec, batch):
    """One measured stage with Q = diag(0, Q_w): P_1 = 0, so w_1 = -Q_w^{-1} l_w and w_0 = -P~0^{-1}^{-1} l_x.
    Bound: numpy's substitutions in the same precision on the same systems, times 8 for the order of the sums."""
    import torch
    dt = np.float64 if prec == mhe.MHE_FP64 else np.float32
    scale = 1e10 if prec == mhe.MHE_FP64 else 1e4
    rng = np.random.default_rng(n + m)
    leaf = [_stiff(rng, m, scale, dt) for _ in range(batch)]
    first = [_stiff(rng, n, scale, dt) for _ in range(batch)]
    nq = n + m
    Q, l = np.zeros((batch, nq, nq)), np.zeros((batch, nq))
    P0 = np.stack([G for G, _ in first])
    for b in range(batch):
        Q[b, n:, n:] = leaf[b][0]
        l[b, n:], l[b, :n] = -leaf[b][1], -first[b][1]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    s = mhe.Solver(n, m, [2] * batch, prec=prec, max_refine=0)
    s.factor(t(0.1 * rng.standard_normal((batch, n, n))), t(0.1 * rng.standard_normal((batch, m, n))), t(Q), t(P0))
    _, w, _ = s.solve(t(l), t(np.zeros((batch, n))), t(np.zeros((batch, n))))
    torch.cuda.synchronize()
    assert np.all(s.infos()["status"] == 0)
    s.close()
    w = w.cpu().numpy().reshape(batch, nq)
    for cases, lo, hi in ((first, 0, n), (leaf, n, nq)):
        got, ref = [], []
        for b, (G, g) in enumerate(cases):
            L = np.linalg.cholesky(G.astype(dt))
            y = solve_triangular(L, g.astype(dt), lower=True)
            ref.append(_residual(G, solve_triangular(L, y, lower=True, trans=1), g))
            got.append(_residual(G, w[b, lo:hi], g))
        assert max(got) <= 8 * max(max(ref), np.finfo(dt).eps), (lo, max(got), max(ref))


@pytest.mark.parametrize("n,m,leaf", [(20, 10, 0), (20, 20, 16)])
def test_mixed_precision_interior_point_iterations(n, m, leaf):
    """Barrier terms make the stages ill-conditioned.  Every Newton step is refined against the FP64 residual, so the
    loop takes FP64's path: half as many iterations again are left for steps that stop at the tolerance."""
    import torch
    Ns = [20 + (37 * i) % 181 for i in range(64)]
    d = device_inputs([synth.mhe_instance(7100 + i, n, m, m, N) for i, N in enumerate(Ns)])
    lo = torch.full((len(Ns), m), -1.0, dtype=torch.float64, device="cuda")
    taken = {}
    for prec in (mhe.MHE_FP64, mhe.MHE_FP32_IR):
        s = mhe.Solver(n, m, Ns, prec=prec, leaf_len=leaf, branching=4 if leaf else 0)
        taken[prec] = s.ip_solve(d["A"], d["B"], d["Q"], d["P0inv"], d["l"], d["a"], d["x0"], lo, -lo)[3]
        s.close()
    assert taken[mhe.MHE_FP32_IR] <= 1.5 * taken[mhe.MHE_FP64], taken
