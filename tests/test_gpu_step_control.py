"""The persistent step kernel outside a plain solve: replayed passes, waits that run out, and the per-pass kernels in
its place (needs a GB300)."""
import numpy as np
import pytest

import lpgen
from tests.test_gpu_parity import ITER_TOL, rel_err
from tests.test_gpu_steps import CASES

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


def _device_error(f, *a, **kw):
    with pytest.raises(P.PdhgcError) as e:
        f(*a, **kw)
    assert e.value.code == -10


def _results(g):
    return [*g.get_solution(P.PHASE1), *g.get_solution(P.CORNER), *(g.get_iterates()[k] for k in ("x", "y"))]


# flow order, flow order with hot copies, barrier order; a few tens of CTAs or more each: two that run in step may
# never find a value missing
ORDERS = {"flow": lambda: lpgen.small_face_lp(2), "hot": CASES["hot_lengths"], "barrier": CASES["barrier_order"]}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", list(ORDERS))
def test_a_wait_that_runs_out_is_reported_by_its_own_call(name, precision):
    """Failure detection without a fault: waits that give up at once make the solve, the corner phase, a restored
    state and (in barrier order) the replayed passes return DEVICE; the next call gives the handle's usual bits."""
    lp = ORDERS[name]()
    kw = dict(max_iters=256, eps_rel=-1.0, algorithm=P.HALPERN,
              precision=P.FP64 if precision == "fp64" else P.FP32_BULK)
    ckw = dict(obj_seed=3, eps_rel=1e30, min_iters=128)
    g = P.lp_from_dict(lp)
    g.solve(**kw)
    state = g.get_state()
    g.corner_phase(**ckw)
    want = _results(g)
    if name == "barrier":
        g.set_wait_limit(0)
        _device_error(g.profile_iteration, 8)
        g.set_wait_limit(1 << 21)
        assert min(g.profile_iteration(8)) > 0
    g.set_wait_limit(0)  # the power iteration's waits
    _device_error(g.solve, **kw)
    _device_error(g.set_state, state)
    g.set_wait_limit(1 << 21)
    g.set_state(state)
    g.solve(**kw)
    g.set_wait_limit(0)
    _device_error(g.corner_phase, **ckw)
    g.set_wait_limit(1 << 21)
    g.corner_phase(**ckw)
    for a, b in zip(_results(g), want):
        assert np.array_equal(a, b)
    g.close()


LOOP = {"hot_lengths": P.LOOP_FLOW, "barrier_order": P.LOOP_BARRIER}  # the others: flow


@pytest.mark.parametrize("algorithm", ["halpern", "averaged"])
@pytest.mark.parametrize("name", list(CASES))
def test_step_kernel_equals_the_per_pass_kernels(name, algorithm):
    """The same phase (a corner phase: 192 iterations, three checks) on a handle that shares the GPU: in FP32 bulk the
    step kernel sums every row in the per-pass kernels' order, so all bits are equal; in FP64 the iterates agree to
    the parity tests' 1e-10."""
    g = P.lp_from_dict(CASES[name]())
    for precision in (P.FP64, P.FP32_BULK):
        g.solve(max_iters=70, eps_rel=-1.0, precision=precision,
                algorithm=P.HALPERN if algorithm == "halpern" else P.AVERAGED)
        out = []
        for shared in (False, True):
            g.set_gpu_sharing(shared)
            assert g.get_loop_kernel(precision) == (P.LOOP_PASSES if shared else LOOP.get(name, P.LOOP_FLOW))
            before = g.kernel_launches()
            rep = g.corner_phase(obj_seed=3, eps_rel=1e30, min_iters=192)
            launches = g.kernel_launches() - before
            it = g.get_iterates()
            out.append((rep["iters"], rep["restarts"], launches, [it[k] for k in ("x", "y", "x_avg", "y_avg")]))
        g.set_gpu_sharing(False)
        (k0, r0, l0, v0), (k1, r1, l1, v1) = out
        assert k0 == k1 == 192 and r0 == r1
        assert l1 - l0 == 192 * 2 - 3  # two launches a step against one per check period
        for a, b in zip(v0, v1):
            if precision == P.FP32_BULK:
                assert np.array_equal(a, b)
            else:
                assert rel_err(a, b) <= ITER_TOL
    g.close()


@pytest.mark.parametrize("algorithm", ["halpern", "averaged"])
def test_handed_off_lps_end_as_on_a_sharing_handle(algorithm):
    """A batch hands an LP off to the single-LP path on the per-pass kernels: the bits of a handle that shares the GPU."""
    lps = [lpgen.small_face_lp(s) for s in range(6)]
    kw = dict(algorithm=P.HALPERN if algorithm == "halpern" else P.AVERAGED)
    B = P.Batch(lps)
    B.set_handoff(16, 128)
    reps = B.solve(**kw)
    handed = [k for k in range(len(lps)) if B.handed_off(k)]
    assert handed
    for k in handed:
        g = P.lp_from_dict(lps[k])
        g.set_gpu_sharing(True)
        rep = g.solve(**kw)
        assert rep["iters"] == reps[k]["iters"] and rep["pobj"] == reps[k]["pobj"] and rep["rel_kkt"] == reps[k]["rel_kkt"]
        g.close()
    B.close()


def test_a_handle_lays_out_the_precision_it_runs_in():
    """Creation launches the two fills of the FP64 step layout and the SELL fills; the FP32 layout's two come with the
    first FP32 solve, whose bits those of later ones are."""
    lp = lpgen.small_face_lp(2)
    g = P.lp_from_dict(lp)
    assert g.kernel_launches() == 2 * 2 + 2
    assert g.get_loop_kernel(P.FP64) == P.LOOP_FLOW and g.get_loop_kernel(P.FP32_BULK) == P.LOOP_PASSES
    kw = dict(max_iters=70, eps_rel=-1.0, algorithm=P.HALPERN)
    counts, xs = [], []
    for precision in (P.FP64, P.FP64, P.FP32_BULK, P.FP32_BULK):
        before = g.kernel_launches()
        g.solve(precision=precision, **kw)
        counts.append(g.kernel_launches() - before)
        xs.append(g.get_iterates()["x"])
    assert counts[0] == counts[1] and counts[2] == counts[3] + 2
    assert np.array_equal(xs[0], xs[1]) and np.array_equal(xs[2], xs[3])
    assert g.get_loop_kernel(P.FP32_BULK) == P.LOOP_FLOW
    g.close()
