"""The ways a solve can be launched give the same result: a small batch in one launch
(a cluster of CTAs per instance), a larger one pass by pass with the last corrections in one
launch, and levels of many chunks (one team of the shape's width per chunk) or few (wider
teams).  Timing marks want a launch per pass, so a context with timing enabled takes the
pass-by-pass route: same kernels' arithmetic, hence equal bits."""
import numpy as np
import pytest

import oracle
from paper_1510_03110_gb300 import mhe, synth
from gpu_util import device_inputs, rel_err, split

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (2, 1), (3, 2), (4, 2), (6, 3), (12, 6), (20, 10), (24, 12)]


def _run(d, form, prec, timing, **kw):
    import torch
    n, m = d["n"], d["m"]
    s = mhe.Solver(n, m, d["N"], prec=prec, **kw)
    if timing:
        mhe.mhe_timing_enable(s.ctx)
    if form == "estimate":
        out = s.estimate(d["q"], d["A"], d["B"], d["C"], d["R"], d["a"], d["yt"], d["wt"], d["x0"], d["P0inv"])
    else:
        s.factor(d["A"], d["B"], d["Q"], d["P0inv"])
        out = s.solve(d["l"], d["a"], d["x0"])
    torch.cuda.synchronize()
    info = s.infos().copy()
    launches = mhe.mhe_launch_count(s.ctx)
    s.close()
    return out, info, launches


def _same(a, b):
    import torch
    for x, y in zip(a[0], b[0]):
        assert torch.equal(x, y)
    for f in ("status", "refine_iters", "relres", "est_relerr"):
        assert np.array_equal(a[1][f], b[1][f]), f


@pytest.mark.parametrize("n,m", SHAPES)
@pytest.mark.parametrize("form,prec,tol", [("solve", mhe.MHE_FP64, 0.0), ("solve", mhe.MHE_FP32_IR, 1e-12),
                                           ("estimate", mhe.MHE_FP32_IR, 1e-12)])
def test_one_launch_equals_pass_by_pass(n, m, form, prec, tol):
    # one long instance (the largest cluster), horizons at the edges of chunks and of a team's share,
    # and enough instances for clusters of one CTA
    for Ns in ([130], [1, 2, 3, 9, 33], [7 + i % 30 for i in range(100)]):
        insts = [synth.mhe_instance(4100 + i, n, m, m, N) for i, N in enumerate(Ns)]
        d = device_inputs(insts)
        a = _run(d, form, prec, False, refine_tol=tol, max_refine=6)
        b = _run(d, form, prec, True, refine_tol=tol, max_refine=6)
        _same(a, b)
        assert a[2] < b[2]   # and it did take the single launch


@pytest.mark.parametrize("n,m,form,tol", [(6, 3, "estimate", 1e-16), (12, 6, "solve", 1e-18),
                                          (24, 12, "estimate", 1e-16)])
def test_last_corrections_in_one_launch(n, m, form, tol):
    # a tolerance at the rounding level (some instances stop early, some use every correction), and one
    # below it (the FP64 Q-form residual meets 1e-16 within four)
    Ns = [2 + (7 * i) % 45 for i in range(260)]
    insts = [synth.mhe_instance(4300 + i, n, m, m, N) for i, N in enumerate(Ns)]
    d = device_inputs(insts)
    a = _run(d, form, mhe.MHE_FP32_IR, False, refine_tol=tol, max_refine=9)
    b = _run(d, form, mhe.MHE_FP32_IR, True, refine_tol=tol, max_refine=9)
    _same(a, b)
    assert a[1]["refine_iters"].max() > 5   # past the change-over


@pytest.mark.parametrize("form", ["solve", "estimate"])
@pytest.mark.parametrize("n,m,Ns,resumed", [
    (6, 3, [2 + (37 * i) % 290 for i in range(180)], True),
    (12, 6, [2 + (37 * i) % 290 for i in range(180)], True),
    (20, 10, [2 + (7 * i) % 60 for i in range(200)], True),
    (20, 10, [1500], True), (24, 12, [900, 5], True),                   # a long horizon, alone or nearly
    (12, 6, [2 + (37 * i) % 290 for i in range(320)], True),            # many instances of longer stages
    (20, 10, [4500], False), (12, 6, [9000, 3], False)])                # horizons too long for sixteen CTAs
def test_late_corrections_take_the_route_of_the_rule(n, m, Ns, resumed, form):
    """More than four corrections: the rest in one launch, or pass by pass to the end; equal bits either way."""
    insts = [synth.mhe_instance(4400 + i % 40, n, m, m, N) for i, N in enumerate(Ns)]
    d = device_inputs(insts)
    a = _run(d, form, mhe.MHE_FP32_IR, False, refine_tol=1e-30, max_refine=9)
    b = _run(d, form, mhe.MHE_FP32_IR, True, refine_tol=1e-30, max_refine=9)
    _same(a, b)
    assert a[1]["refine_iters"].max() == 9
    assert (a[2] < b[2]) if resumed else (a[2] == b[2]), (a[2], b[2])


@pytest.mark.parametrize("n,m", [(4, 2), (6, 3), (12, 6), (20, 10), (24, 12)])
@pytest.mark.parametrize("prec,tol", [(mhe.MHE_FP64, 1e-10), (mhe.MHE_FP32_IR, 1e-8)])
def test_levels_of_many_chunks(n, m, prec, tol):
    """More level-0 chunks than the wider teams take (1216): the shape's own team, against the oracle."""
    Ns = [(2, 5, 9, 17, 30)[i % 5] for i in range(640)]
    insts = [synth.mhe_instance(4500 + i, n, m, m, N) for i, N in enumerate(Ns)]
    d = device_inputs(insts)
    out, info, _ = _run(d, "solve", prec, False, leaf_len=4 if n <= 4 else 8, branching=2, top_len=2,
                        refine_tol=1e-13 if prec == mhe.MHE_FP32_IR else 0.0, max_refine=8)
    assert np.all(info["status"] == 0)
    sols = split(*out, Ns, n, m)
    for b in list(range(5)) + [317, 638, 639]:
        ref = oracle.riccati(oracle.mhe_to_uftoc(insts[b]))
        assert rel_err(sols[b], ref) <= tol, (b, Ns[b])


@pytest.mark.parametrize("n,m", [(6, 3), (12, 6)])
def test_master_levels_of_many_chunks(n, m):
    """More chunks than the wider teams take (1216) at a master level too, FP64: the shape's own team, against the oracle."""
    Ns = [34] * 640
    insts = [synth.mhe_instance(4600 + i % 64, n, m, m, N) for i, N in enumerate(Ns)]
    d = device_inputs(insts)
    s = mhe.Solver(n, m, Ns, prec=mhe.MHE_FP64, leaf_len=8, branching=2, top_len=2)
    assert mhe.mhe_plan_info(s.ctx)[1][1] > 1216
    s.close()
    out, info, _ = _run(d, "solve", mhe.MHE_FP64, False, leaf_len=8, branching=2, top_len=2)
    assert np.all(info["status"] == 0)
    sols = split(*out, Ns, n, m)
    for b in (0, 1, 63, 317, 639):
        assert rel_err(sols[b], oracle.riccati(oracle.mhe_to_uftoc(insts[b]))) <= 1e-10, b


def test_preparation_of_zeros_and_extreme_entries():
    """Entries that leave the fast conversion (zeros, tiny and huge magnitudes) against the FP64 solution."""
    n, m = 6, 3
    insts = [synth.mhe_instance(4700 + i, n, m, m, 20) for i in range(3)]
    for p in insts:
        p["A"][:, 0, :] = 0.0
        p["A"][:, 1, 2] = 1e-42
        p["B"][:, 2, 1] = -1e-300
        p["C"][:, 0, 0] = 0.0
        p["a"][:] *= 1e6
    d = device_inputs(insts)
    out, info, _ = _run(d, "estimate", mhe.MHE_FP32_IR, False, refine_tol=1e-13, max_refine=8)
    assert np.all(info["status"] == 0)
    for sol, p in zip(split(*out, d["N"], n, m), insts):
        assert rel_err(sol, oracle.riccati(oracle.mhe_to_uftoc(p))) <= 1e-8


@pytest.mark.parametrize("first_only", [True, False])
def test_whole_instances_on_the_tensor_cores(first_only):
    """nx = 64, TF32 products, plans of one level: more instances than two teams an SM, horizons from the arrival
    stage alone up; factors kept for another right-hand side.  The first solve's error against FP32's:
    the split products are as accurate as an FP32 chain (2.0e-7 against 1.8e-7 of sum |ab|), everything
    after them is the same arithmetic in another order; a factor 8 is left for the order."""
    n, m = 64, 32
    Ns = [1 + i % 4 for i in range(320)] + [33]
    insts = [synth.mhe_instance(4900 + i % 24, n, m, m, N) for i, N in enumerate(Ns)]
    d = device_inputs(insts)
    err = {}
    for prec in (mhe.MHE_TF32_IR, mhe.MHE_FP32_IR):
        out, info, _ = _run(d, "solve", prec, False, top_len=1000, refine_tol=1e-13,
                            max_refine=0 if first_only else 20)
        sols = split(*out, Ns, n, m)
        for b in list(range(4)) + [303, 304, 319, 320]:
            e = rel_err(sols[b], oracle.riccati(oracle.mhe_to_uftoc(insts[b])))
            err[prec, b] = e
            if not first_only:
                assert info["status"][b] == 0 and e <= 1e-8, (prec, b, e, info[b])
    if first_only:
        most = {p: max(e for (q, _), e in err.items() if q == p) for p in (mhe.MHE_TF32_IR, mhe.MHE_FP32_IR)}
        assert most[mhe.MHE_TF32_IR] <= 8 * most[mhe.MHE_FP32_IR], most


@pytest.mark.parametrize("where", [0, 1, 4])
def test_failed_pivot_of_a_whole_instance_on_the_tensor_cores(where):
    """The failed stage (the arrival stage, the first and the last measured one) is reported for its instance only."""
    n, m, N = 64, 32, 5
    insts = [synth.mhe_instance(5000 + i, n, m, m, N) for i in range(3)]
    d = device_inputs(insts)
    if where == 0:
        d["P0inv"].view(3, n * n)[1].mul_(-1e6)
    else:
        import torch
        q = d["Q"].view(3, N - 1, n + m, n + m)[1, where - 1]
        q[n:, n:] = -1e6 * torch.eye(m, dtype=torch.float64, device="cuda")
    _, info, _ = _run(d, "solve", mhe.MHE_TF32_IR, False, top_len=1000, refine_tol=1e-12, max_refine=4)
    assert info["status"][1] == -3 and info["stage"][1] == where and info["chunk"][1] == 1, info[1]
    assert info["status"][0] == 0 and info["status"][2] == 0
