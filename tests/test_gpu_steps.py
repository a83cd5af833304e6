"""The persistent step kernel (csrc/steps.cuh) against the oracle at the sizes
where its layout and its two orders (flow, barrier) can go wrong: single rows
and columns, units of 31 to 33 rows, empty rows and columns, rows at the hot
length, rows cut into parts, barrier-order sizes (needs a GB300).

FP64: iterates after 70 steps (one check, and an incomplete second chunk) to
the parity tests' 1e-10.  FP32 bulk: each of the 70 x 2 passes rounds matrix
values and gathered entries to 2^-24; over a row of `len` entries that grows as
sqrt(len), is scaled by at most max(omega, 1 / omega) (the step sizes are
eta omega^(+-1) with eta |A_hat| < 1), and is relative to the larger iterate.
"""
import numpy as np
import pytest

import lpgen
import oracle
from tests.test_gpu_parity import ITER_TOL, rel_err

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2511_13894_gb300.pdhgc")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

FP32_STEPS = 70 * 2 * 2.0 ** -24


def _lp(m, n, row_len, seed, full_cols=0, empty=()):
    """Rows of length row_len(i) with random columns (the first full_cols columns in every row), '<' rows, boxes."""
    r = np.random.default_rng(seed)
    cols, rp = [], [0]
    for i in range(m):
        k = 0 if i in empty else min(n, row_len(i))
        c = np.zeros(0, np.int64)
        if k:
            rest = r.choice(np.arange(full_cols, n), size=max(0, k - full_cols), replace=False) if n > full_cols else []
            c = np.concatenate([np.arange(min(full_cols, k)), rest]).astype(np.int64)
        cols.append(c)
        rp.append(rp[-1] + len(c))
    col = np.concatenate(cols).astype(np.int32)
    val = r.standard_normal(len(col))
    x = r.uniform(0.0, 2.0, n)
    ax = np.array([val[rp[i]:rp[i + 1]] @ x[col[rp[i]:rp[i + 1]]] for i in range(m)])
    sense = r.choice(np.array([lpgen.EQ, lpgen.LE], dtype=np.int8), size=m)
    return dict(m=m, n=n, row_ptr=np.array(rp, dtype=np.int64), col_idx=col, val=val,
                b=ax + np.where(sense == lpgen.LE, 0.5, 0.0), c=r.standard_normal(n), lb=np.zeros(n),
                ub=np.where(r.random(n) < 0.5, 3.0, np.inf), sense=sense)


CASES = {
    "one_entry": lambda: _lp(1, 1, lambda i: 1, 1),
    "one_row_of_33": lambda: _lp(1, 33, lambda i: 33, 2),
    "31_rows": lambda: _lp(31, 65, lambda i: 1 + i % 7, 3, empty=(4, 30)),
    "33_rows_32_columns": lambda: _lp(33, 32, lambda i: 1 + i % 5, 4),
    "hot_lengths": lambda: _lp(260, 700, lambda i: 126 + i % 5, 5, full_cols=2),
    "split_rows": lambda: _lp(40, 3000, lambda i: 3000 if i < 2 else 9 + 61 * (i % 3), 6, full_cols=1),
    "barrier_order": lambda: _lp(500, 2100, lambda i: 100 + i % 67, 7, full_cols=3),
}


@pytest.mark.parametrize("algorithm", ["halpern", "averaged"])
@pytest.mark.parametrize("name", list(CASES))
def test_step_kernel_matches_oracle(name, algorithm):
    lp = CASES[name]()
    ref = oracle.run_iterations(lp, 70, dict(algorithm=algorithm))
    s = ref["state"]
    second = (s.xp, s.yp) if algorithm == "halpern" else s.average()
    g = P.lp_from_dict(lp)
    longest = max(np.diff(lp["row_ptr"]).max(), np.bincount(lp["col_idx"]).max())
    scale = max(1.0, np.abs(s.x).max(), np.abs(s.y).max())
    tol32 = FP32_STEPS * scale * np.sqrt(longest) * max(s.omega, 1.0 / s.omega)
    for precision, tol in ((P.FP64, ITER_TOL), (P.FP32_BULK, tol32)):
        # twice: the step numbers of the second solve continue the first's
        for _ in range(2):
            rep = g.solve(max_iters=70, eps_rel=-1.0, precision=precision,
                          algorithm=P.HALPERN if algorithm == "halpern" else P.AVERAGED)
            assert rep["status_name"] == "ITER_LIMIT" and rep["iters"] == 70
            it = g.get_iterates()
            assert it["restarts"] == s.restarts
            for got, want in ((it["x"], s.x), (it["y"], s.y), (it["x_avg"], second[0]), (it["y_avg"], second[1])):
                assert rel_err(got, want) <= tol, precision
        assert abs(g.get_scaling()["sigma_max"] - ref["sigma_max"]) <= 1e-12 * max(1.0, ref["sigma_max"])
    g.close()


def test_profiled_passes_leave_the_solver_sound():
    """The timed single passes write no step number that a later solve could wait for."""
    lp = lpgen.small_face_lp(2)
    g = P.lp_from_dict(lp)
    g.solve(max_iters=128, eps_rel=-1.0, algorithm=P.HALPERN)
    x = g.get_iterates()["x"]
    ms = g.profile_iteration(100)
    assert len(ms) == 2 and min(ms) > 0
    g.solve(max_iters=128, eps_rel=-1.0, algorithm=P.HALPERN)
    assert np.array_equal(g.get_iterates()["x"], x)
    g.close()
