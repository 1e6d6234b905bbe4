"""The residual norm behind mhe_info.relres is taken in 64 bits where the rows are computed in 64
bits: the arrival stage of the double-float residual.  Instances of one (arrival) stage and no
corrections: the FP32 solution's rows are exact in FP64 (sums and differences of a float and a
double of like size), so relres is reproducible to a few roundings of its own quotient."""
import numpy as np
import pytest

from paper_1510_03110_gb300 import mhe, synth
from gpu_util import device_inputs, split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(2, 1), (4, 2), (6, 3), (12, 6), (20, 10), (24, 12), (64, 32)])
@pytest.mark.parametrize("timing", [False, True])   # the one-launch solve, and a launch per pass
def test_arrival_rows_enter_the_norm_in_64_bits(n, m, timing):
    import torch
    # (a last instance with measured stages: without any the MHE form has no C and R)
    insts = [synth.mhe_instance(5200 + i, n, m, m, 1) for i in range(9)] + [synth.mhe_instance(5299, n, m, m, 3)]
    d = device_inputs(insts)
    s = mhe.Solver(n, m, d["N"], prec=mhe.MHE_FP32_IR, refine_tol=1e-30, max_refine=0)
    if timing:
        mhe.mhe_timing_enable(s.ctx)
    out = s.estimate(m, d["A"], d["B"], d["C"], d["R"], d["a"], d["yt"], d["wt"], d["x0"], d["P0inv"])
    torch.cuda.synchronize()
    info = s.infos()
    s.close()
    for sol, p, o in list(zip(split(*out, d["N"], n, m), insts, info))[:-1]:
        x, w, lam = sol["x"], sol["w"], sol["lam"]
        rows = np.concatenate([p["x0"] - x[0], lam[1] - lam[0], p["P0inv"] @ w + lam[1], x[0] + w - x[1], lam[1]])
        z = max(np.abs(x).max(), np.abs(w).max(), np.abs(lam).max())
        assert np.array_equal(p["P0inv"], np.eye(n))   # ||K|| = 3: the dynamics rows
        ref = np.abs(rows).max() / (3.0 * z + np.abs(p["x0"]).max())
        assert ref > 0 and abs(o["relres"] - ref) <= 4 * 2.0 ** -53 * ref, (o["relres"], ref)
