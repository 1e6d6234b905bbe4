"""The work this library is measured on: MHE Newton steps through its public entry points.

Every case is a call a program makes in earnest (`Solver.factor_solve`, `Solver.solve`,
`Solver.estimate`, `Server.submit` / `Server.wait`) on synthetic MHE problems of the
construction the benchmark uses (`paper_1510_03110_gb300/synth.py`): per stage
A = 0.95 A_raw / rho(A_raw), B, C ~ N(0, 1), R = M M^T + 0.1 I, offsets ~ N(0, 1), P~0 = I.
The stages are drawn on the GPU, each stage its own, and rho(A_raw) comes from repeated
squaring (Gelfand's formula), to well within a percent.

The families (`kind`):
  newton    one factorisation and solve of a UFTOC problem (A, B, Q, l given), as inside an
            optimisation loop
  resolve   a new right-hand side on a factorisation the program keeps
  estimate  the whole step from MHE data (stage assembly included)
  serve     receding-horizon estimators on a server: one new sample for each, every answer awaited
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1510_03110_gb300 import mhe

PREC = {"fp64": mhe.MHE_FP64, "fp32": mhe.MHE_FP32_IR, "tf32": mhe.MHE_TF32_IR}


def _case(name, kind, nx, batch, n_lo, n_hi, prec, leaf=0, branching=0, serial=False, graph=False, tol=0.0, refine=-1):
    """nw = ny = nx / 2; horizons uniform in [n_lo, n_hi]; leaf, branching 0 = the library's defaults."""
    return dict(name=name, kind=kind, nx=nx, batch=batch, n_lo=n_lo, n_hi=n_hi, prec=prec, leaf=leaf,
                branching=branching, serial=serial, graph=graph, tol=tol, refine=refine)


def listed():
    return [
        # the correctness and latency configuration: one small plant, FP64, a Newton step at a time
        _case("newton_nx4_N64_fp64", "newton", 4, 1, 64, 64, "fp64", leaf=4, branching=2),
        # one estimator's sample instant in a real-time loop: fixed buffers, replayed as a graph
        _case("tick_nx12_N200_graph", "estimate", 12, 1, 200, 200, "fp32", graph=True, tol=TOL, refine=16),
        # the same without replay for a larger plant and a long window (a program whose buffers change)
        _case("tick_nx24_N1000", "estimate", 24, 1, 1000, 1000, "fp32", tol=TOL, refine=16),
        # single horizons of the paper's depth experiment (nx = 20), FP64: moderate and long
        _case("horizon_nx20_N1024_fp64", "newton", 20, 1, 1024, 1024, "fp64", leaf=16, branching=4),
        _case("horizon_nx20_N16384_fp64", "newton", 20, 1, 16384, 16384, "fp64", leaf=32, branching=4),
        # a bank of plants solved in FP64, as the inner step of the box-bounded interior-point loop
        _case("bank_nx12_fp64", "newton", 12, 256, 32, 512, "fp64", leaf=16, branching=4),
        # the same bank with the factorisation kept: a new right-hand side, mixed precision
        _case("resolve_nx12_fp32", "resolve", 12, 256, 32, 512, "fp32", leaf=16, branching=4, tol=TOL, refine=16),
        # the batched uneven workload's three shapes (plans as its autotuner chose them)
        _case("batch_nx6", "estimate", 6, 1024, 32, 2048, "fp32", leaf=32, branching=4, tol=TOL, refine=16),
        _case("batch_nx12", "estimate", 12, 1024, 32, 2048, "fp32", leaf=64, branching=4, tol=TOL, refine=16),
        _case("batch_nx24", "estimate", 24, 512, 32, 2048, "fp32", leaf=128, branching=4, tol=TOL, refine=16),
        # large states, tensor-core stage products, every instance one chunk (the autotuner's choice)
        _case("batch_nx64_tf32", "estimate", 64, 256, 512, 512, "tf32", serial=True, tol=TOL, refine=16),
        # a server's sample instant: 64 estimators, windows of 200, factorisations reused across the shift
        _case("serve_nx12_N200", "serve", 12, 64, 200, 200, "fp32", tol=TOL, refine=16),
    ]


# refinement target of the mixed-precision cases.  At the benchmark's 1e-12 single entries of the
# worst-conditioned instances (nx = 24, long horizons) are 4e-8 off; a program that wants every entry
# to 1e-8, the accuracy the library's own tests ask of a refined solve, asks for one digit more.
TOL = 1e-13


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case of the same families: sizes log-uniform over the listed ranges."""
    kind = rng.choice(["single", "horizon", "bank", "resolve", "batch", "batch", "xl", "serve"])
    if kind == "single":
        nx = rng.choice([4, 6, 12, 24])
        N = _log(rng, 33, 1000)
        c = _case("", "estimate", nx, 1, N, N, "fp32", graph=rng.random() < 0.5, tol=TOL, refine=16)
    elif kind == "horizon":
        nx = rng.choice([4, 12, 20])
        N = _log(rng, 64, 16384)
        c = _case("", "newton", nx, 1, N, N, "fp64", leaf=rng.choice([8, 16, 32]), branching=4)
    elif kind in ("bank", "resolve"):
        nx = rng.choice([4, 6, 12, 20])
        hi = _log(rng, 50, 512)
        c = _case("", "newton" if kind == "bank" else "resolve", nx, _log(rng, 8, 256), 32, hi,
                  "fp64" if kind == "bank" else "fp32", leaf=16, branching=4, tol=0.0 if kind == "bank" else TOL,
                  refine=-1 if kind == "bank" else 16)
    elif kind == "batch":
        nx = rng.choice([6, 12, 24])
        leaf = {6: 32, 12: 64, 24: 128}[nx]
        c = _case("", "estimate", nx, _log(rng, 32, 512 if nx == 24 else 1024), 32, _log(rng, 200, 2048), "fp32",
                  leaf=leaf, branching=4, tol=TOL, refine=16)
    elif kind == "serve":
        N = _log(rng, 50, 200)
        c = _case("", "serve", rng.choice([6, 12, 24]), _log(rng, 8, 64), N, N, "fp32", tol=TOL, refine=16)
    else:
        N = _log(rng, 100, 512)
        c = _case("", "estimate", 64, _log(rng, 40, 256), N, N, "tf32", serial=True, tol=TOL, refine=16)
    del c["name"]
    return c


def _horizons(case):
    """The horizons of the batch: part of the plan, so of the case and not of the seed."""
    if case["n_lo"] == case["n_hi"]:
        return np.full(case["batch"], case["n_lo"], dtype=np.int64)
    return np.random.default_rng([7, case["nx"], case["batch"], case["n_hi"]]).integers(case["n_lo"], case["n_hi"] + 1, size=case["batch"])


def _spectral_radius(A):
    """rho of every matrix of the stack: ||A^1024||^(1/1024) by ten squarings, rescaled as they go."""
    X = A.float()
    log = torch.zeros(A.shape[0], dtype=torch.float64, device=A.device)
    for k in range(11):
        s = X.flatten(1).norm(dim=1).clamp_min(1e-30)
        X = X / s[:, None, None]
        log += s.double().log() / 2.0 ** k
        if k < 10:
            X = X @ X
    return log.exp()


def _mhe_data(case, seed, S, batch):
    """S stages and `batch` arrival states on the GPU: every matrix a column-major block per row."""
    n, m = case["nx"], case["nx"] // 2
    q = m
    g = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + n)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)

    A = normal(S, n, n)
    for i in range(0, S, 1 << 16):   # in pieces: bounded scratch memory
        Ai = A[i:i + (1 << 16)]
        Ai *= (0.95 / _spectral_radius(Ai))[:, None, None]
    B = normal(S, m, n)
    C = normal(S, n, q)
    M = normal(S, m + q, m + q)
    R = M @ M.transpose(1, 2)
    R.diagonal(dim1=1, dim2=2).add_(0.1)
    del M
    d = dict(A=A.reshape(S, -1), B=B.reshape(S, -1), C=C.reshape(S, -1), R=R.reshape(S, -1), a=normal(S, n),
             yt=normal(S, q), wt=normal(S, m), x0=normal(batch, n))
    d["P0inv"] = torch.eye(n, dtype=torch.float64, device="cuda").expand(batch, n, n).reshape(batch, -1).contiguous()
    return d


def _cols(t, r, c):
    """Column-major blocks as a stack of r x c matrices (a view)."""
    return t.reshape(-1, c, r).transpose(1, 2)


def _uftoc(d, n, m, q):
    """Q_t and l_t of every stage, plain torch (Section II of the paper)."""
    C, R = _cols(d["C"], q, n), _cols(d["R"], m + q, m + q)
    W, S, V = R[:, :m, :m], R[:, :m, m:], R[:, m:, m:]
    y, w = d["yt"][:, :, None], d["wt"][:, :, None]
    Q = torch.empty(C.shape[0], n + m, n + m, dtype=torch.float64, device=C.device)
    Q[:, :n, :n] = C.transpose(1, 2) @ (V @ C)
    Q[:, :n, :n] = 0.5 * (Q[:, :n, :n] + Q[:, :n, :n].transpose(1, 2))
    SC = S @ C
    Q[:, n:, :n] = -SC
    Q[:, :n, n:] = -SC.transpose(1, 2)
    Q[:, n:, n:] = W
    l = torch.cat([C.transpose(1, 2) @ (S.transpose(1, 2) @ w - V @ y), S @ y - W @ w], dim=1)[:, :, 0]
    return Q, l


def _server_data(case, seed):
    """Host data of the estimators: N - 1 stages of the first window and a cycle of new samples each."""
    n, m, E, N = case["nx"], case["nx"] // 2, case["batch"], case["n_lo"]
    L = N - 1 + 16
    d = _mhe_data(case, seed, E * L, E)
    host = {k: v.cpu().numpy() for k, v in d.items()}
    return d, host, L


def prepare(case, seed):
    n, m = case["nx"], case["nx"] // 2
    q = m
    if case["kind"] == "serve":
        E, N = case["batch"], case["n_lo"]
        _, h, L = _server_data(case, seed)
        srv = mhe.Server(8 << 30, prec=PREC[case["prec"]], refine_tol=case["tol"], max_refine=case["refine"])
        ids, samples = [], []
        for e in range(E):
            def blocks(key, r, c):
                return h[key][e * L:(e + 1) * L].reshape(L, c, r).transpose(0, 2, 1)
            st = dict(A=blocks("A", n, n), B=blocks("B", n, m), C=blocks("C", q, n), R=blocks("R", m + q, m + q),
                      **{k: h[k][e * L:(e + 1) * L] for k in ("a", "yt", "wt")})
            ids.append(srv.open(dict(n=n, m=m, q=q, N=N, x0=h["x0"][e], P0inv=np.eye(n),
                                     **{k: v[:N - 1] for k, v in st.items()})))
            samples.append([mhe.pack_stage(*(st[k][j] for k in ("A", "B", "C", "R", "a", "yt", "wt")))
                            for j in range(N - 1, L)])
        return dict(kind="serve", srv=srv, ids=ids, samples=samples, tick=0, n=n)
    N = _horizons(case)
    S, batch = int(np.sum(N - 1)), case["batch"]
    d = _mhe_data(case, seed, S, batch)
    # a graph is captured on a stream of the program's own
    stream = torch.cuda.Stream() if case["graph"] else None
    s = mhe.Solver(n, m, N, prec=PREC[case["prec"]], leaf_len=case["leaf"], branching=case["branching"],
                   top_len=int(N.max()) + 1 if case["serial"] else 0, refine_tol=case["tol"],
                   max_refine=case["refine"], stream=stream)
    if case["graph"]:
        s.set_graph(True)
    state = dict(kind=case["kind"], s=s, out=s.outputs(), q=q)
    if case["kind"] == "estimate":
        state["data"] = [d[k] for k in ("A", "B", "C", "R", "a", "yt", "wt", "x0", "P0inv")]
    else:
        Q = torch.empty(max(1, S), (n + m) ** 2, dtype=torch.float64, device="cuda")
        l = torch.empty(max(1, S), n + m, dtype=torch.float64, device="cuda")
        mhe.mhe_assemble(n, m, q, d["C"], d["R"], d["yt"], d["wt"], Q, l)
        state["mats"] = [d["A"], d["B"], Q, d["P0inv"]]
        state["rhs"] = [l, d["a"], d["x0"]]
        if case["kind"] == "resolve":
            s.factor(*state["mats"])
    torch.cuda.synchronize()   # the solver's stream may be another than the one that made the inputs
    return state


def run(state):
    if state["kind"] == "serve":
        srv, n = state["srv"], state["n"]
        k = state["tick"] = state["tick"] + 1
        tickets = [srv.submit(i, smp[(k - 1) % len(smp)]) for i, smp in zip(state["ids"], state["samples"])]
        return np.stack([srv.wait(t, n)["x"] for t in tickets])
    s = state["s"]
    if state["kind"] == "estimate":
        return s.estimate(state["q"], *state["data"], out=state["out"])
    if state["kind"] == "resolve":
        return s.solve(*state["rhs"], out=state["out"])
    return s.factor_solve(*state["mats"], *state["rhs"], out=state["out"])


def _stages(case):
    return int(np.sum(_horizons(case) - 1))


def work(case):
    n, m = case["nx"], case["nx"] // 2
    q = m
    S, batch = _stages(case), case["batch"]
    solution = (S + 2 * batch) * 2 * n + S * m + batch * n
    # Algorithms 1-3: P [A B], A^T P A and B^T P B (symmetric), A^T P B, chol G, K, P - H K (symmetric), the vectors
    factor = 2 * n * n * (n + m) + n ** 3 + n * m * m + 2 * n * n * m + m ** 3 / 3 + 2 * n * m * m + n * n * m
    solve = 2 * (2 * n * n + 2 * n * m + n * m) + 2 * (n * n + 2 * n * m) + 2 * n * n + 2 * m * m
    if case["kind"] == "serve":
        stage = n * n + n * m + q * n + (m + q) ** 2 + n + q + m
        # one new stage in and one answer out per estimator; the right-hand side of every window again
        return dict(bytes=8.0 * batch * (stage + n) + 4.0 * S * (2 * n * n + 3 * n * m), flops=float(S * solve + batch * factor))
    rhs = S * (n + m + n) + batch * n
    if case["kind"] == "resolve":
        mats = S * (n * n + n * m + m * m + m * n) * (1 if case["prec"] == "fp64" else 0.5)
        return dict(bytes=8.0 * (mats + rhs + solution), flops=float(S * solve))
    if case["kind"] == "newton":
        mats = S * (n * n + n * m + (n + m) ** 2) + batch * n * n
        return dict(bytes=8.0 * (mats + rhs + solution), flops=float(S * (factor + solve)))
    data = S * (n * n + n * m + q * n + (m + q) ** 2 + n + q + m) + batch * (n * n + n)
    assemble = 2 * q * q * n + 2 * m * q * n + n * n * q
    return dict(bytes=8.0 * (data + solution), flops=float(S * (factor + solve + assemble)))


def _riccati(A, B, Q, l, a, x0, P0inv, N):
    """The Newton step by the serial Riccati recursion, batched over the instances, in FP64.

    A, B, Q, l, a: the caller's stages, instance after instance (matrix stacks); returns x, w, lam
    in the library's layout."""
    dev, n, m, nb = A.device, A.shape[1], B.shape[2], len(N)
    order = np.argsort(-N, kind="stable")
    off = np.concatenate([[0], np.cumsum(N - 1)[:-1]])[order]
    Ns = N[order]
    alive = [int(np.searchsorted(-Ns, -t, side="left")) for t in range(int(Ns[0]) + 1)]   # instances with N > t
    offd = torch.as_tensor(off, device=dev)
    P = torch.zeros(nb, n, n, dtype=torch.float64, device=dev)
    Psi = torch.zeros(nb, n, 1, dtype=torch.float64, device=dev)
    Ks = torch.empty(A.shape[0], m, n, dtype=torch.float64, device=dev)
    ks = torch.empty(A.shape[0], m, 1, dtype=torch.float64, device=dev)
    Ps = torch.empty(A.shape[0], n, n, dtype=torch.float64, device=dev)
    Psis = torch.empty(A.shape[0], n, 1, dtype=torch.float64, device=dev)

    def gains(G, H, g):
        L = torch.linalg.cholesky_ex(G)[0]
        Y = torch.linalg.solve_triangular(L, torch.cat([H.transpose(1, 2), g], dim=2), upper=False)
        X = torch.linalg.solve_triangular(L.transpose(1, 2), Y, upper=True)
        return Y[:, :, :n], -X[:, :, :n], X[:, :, n:]

    for t in range(int(Ns[0]) - 1, 0, -1):
        k = alive[t]
        s = offd[:k] + (t - 1)
        At, Bt, Qt, lt, Pt = A[s], B[s], Q[s], l[s][:, :, None], P[:k]
        PA, PB = Pt @ At, Pt @ Bt
        u = Psi[:k] - Pt @ a[s][:, :, None]
        G = Qt[:, n:, n:] + Bt.transpose(1, 2) @ PB
        H = Qt[:, :n, n:] + At.transpose(1, 2) @ PB
        g = Bt.transpose(1, 2) @ u - lt[:, n:]
        Y, K, kk = gains(0.5 * (G + G.transpose(1, 2)), H, g)
        F = Qt[:, :n, :n] + At.transpose(1, 2) @ PA - Y.transpose(1, 2) @ Y
        P[:k] = 0.5 * (F + F.transpose(1, 2))
        Psi[:k] = At.transpose(1, 2) @ u - lt[:, :n] + K.transpose(1, 2) @ g
        Ks[s], ks[s], Ps[s], Psis[s] = K, kk, P[:k], Psi[:k]
    xo = np.concatenate([[0], np.cumsum(N + 1)[:-1]])[order]
    wo = np.concatenate([[0], np.cumsum(n + (N - 1) * m)[:-1]])[order]
    xod, wod = torch.as_tensor(xo, device=dev), torch.as_tensor(wo, device=dev)
    x = torch.empty(int(np.sum(N + 1)), n, dtype=torch.float64, device=dev)
    lam = torch.zeros_like(x)
    w = torch.empty(int(np.sum(n + (N - 1) * m)), dtype=torch.float64, device=dev)
    # the arrival stage: x_1 = x_0 + w_0, cost 1/2 w_0^T P0inv w_0
    od = torch.as_tensor(order, device=dev)
    x_t = x0[od][:, :, None]
    w0 = torch.linalg.solve(_cols(P0inv, n, n)[od] + P, Psi - P @ x_t)
    x[xod], lam[xod] = x_t[:, :, 0], (P @ (x_t + w0) - Psi)[:, :, 0]
    w[wod[:, None] + torch.arange(n, device=dev)] = w0[:, :, 0]
    x_t = x_t + w0
    for t in range(1, int(Ns[0])):
        k = alive[t]
        s = offd[:k] + (t - 1)
        x_t = x_t[:k]
        x[xod[:k] + t], lam[xod[:k] + t] = x_t[:, :, 0], (Ps[s] @ x_t - Psis[s])[:, :, 0]
        wt = Ks[s] @ x_t + ks[s]
        w[(wod[:k] + n + (t - 1) * m)[:, None] + torch.arange(m, device=dev)] = wt[:, :, 0]
        x_t = A[s] @ x_t + B[s] @ wt + a[s][:, :, None]
        end = Ns[:k] == t + 1
        if end.any():
            e = torch.as_tensor(np.nonzero(end)[0], device=dev)
            x[xod[e] + t + 1] = x_t[e][:, :, 0]
    one = Ns == 1
    if one.any():
        e = torch.as_tensor(np.nonzero(one)[0], device=dev)
        x[xod[e] + 1] = x_t[e][:, :, 0]
    return x, w, lam


def exact(case, seed):
    n, m = case["nx"], case["nx"] // 2
    q = m
    if case["kind"] == "serve":
        # the first pass: the window moved by one sample, the arrival state as given
        E, N = case["batch"], case["n_lo"]
        d, _, L = _server_data(case, seed)
        keep = (torch.arange(E, device="cuda")[:, None] * L + torch.arange(1, N, device="cuda")).reshape(-1)
        d = {k: v if k in ("x0", "P0inv") else v[keep] for k, v in d.items()}
        Ns = np.full(E, N, dtype=np.int64)
        Q, l = _uftoc(d, n, m, q)
        x, _, _ = _riccati(_cols(d["A"], n, n), _cols(d["B"], n, m), Q, l, d["a"], d["x0"], d["P0inv"], Ns)
        return x.reshape(E, N + 1, n)[:, N - 1].cpu().numpy()
    N = _horizons(case)
    d = _mhe_data(case, seed, int(np.sum(N - 1)), case["batch"])
    if case["batch"] == 1:   # one long chain of small products: the host is faster
        d = {k: v.cpu() for k, v in d.items()}
    Q, l = _uftoc(d, n, m, q)
    return _riccati(_cols(d["A"], n, n), _cols(d["B"], n, m), Q, l, d["a"], d["x0"], d["P0inv"], N)
