"""The persistent step kernel outside a plain solve: replayed passes (needs a GB300)."""
import numpy as np
import pytest

import lpgen
from tests.test_gpu_parity import ITER_TOL, rel_err

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2511_13894_gb300.pdhgc")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _replay(lp, sc, it, iters):
    """`iters` primal passes and then as many dual passes of the Halpern loop's first step (weight 1/2, anchor at
    the start point), from the iterates `it`, on the scaled LP in numpy."""
    m, n = lp["m"], lp["n"]
    row = np.repeat(np.arange(m), np.diff(lp["row_ptr"]))
    a = sc["Dr"][row] * lp["val"] * sc["Dc"][lp["col_idx"]]
    lh, uh = lp["lb"] / sc["Dc"], lp["ub"] / sc["Dc"]
    x0 = np.clip(np.zeros(n), lh, uh)
    x, y = it["x"], it["y"]
    g = sc["Dc"] * lp["c"] - np.bincount(lp["col_idx"], a * y[row], n)
    for _ in range(iters):
        xn = np.clip(x - sc["tau"] * g, lh, uh)
        xbar = 2.0 * xn - x
        x = 0.5 * (xbar - x0) + x0
    r = sc["Dr"] * lp["b"] - np.bincount(row, a * xbar[lp["col_idx"]], m)
    for _ in range(iters):
        y = 0.5 * (2.0 * (y + sc["sigma"] * r) - y)
    return x, y


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("iters", [2, 65, 4097, 9000])
def test_replayed_passes_are_steps_inside_a_chunk(iters, precision):
    """Each replayed pass is the chunk's first step (not one of a later weight, nor a check step), whatever
    `iters` is beside the check period (64) and the longest chunk (4096); a later solve keeps its bits."""
    lp = lpgen.small_face_lp(2)
    g = P.lp_from_dict(lp)
    kw = dict(max_iters=32, eps_rel=-1.0, algorithm=P.HALPERN,
              precision=P.FP64 if precision == "fp64" else P.FP32_BULK)
    g.solve(**kw)
    it = g.get_iterates()
    ms = g.profile_iteration(iters)
    assert len(ms) == 2 and min(ms) > 0
    now = g.get_iterates()
    assert np.array_equal(now["x_avg"], it["x_avg"]) and np.array_equal(now["y_avg"], it["y_avg"])
    if precision == "fp64":  # the FP32 loop keeps its own iterates
        x, y = _replay(lp, g.get_scaling(), it, iters)
        assert rel_err(now["x"], x) <= ITER_TOL and rel_err(now["y"], y) <= ITER_TOL
    g.solve(**kw)
    again = g.get_iterates()
    for k in ("x", "y", "x_avg", "y_avg"):
        assert np.array_equal(again[k], it[k]), k
    g.close()
