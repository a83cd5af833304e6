"""What users of this framework have it do, as cases whose passes can be timed.

Each listed case is one kind of use at one size; `draw` spreads the same kinds
over their ranges.  The LPs are those of `lpgen` (the repository's seeded
generators), at the sizes of its named workloads, of its batch and guidance
recipes and between them.  A solve runs a fixed number of iterations instead
of to a tolerance, so that a pass is the same work for every seed: phase 1
stops at its iteration limit, a corner phase at the first check at or after
its minimum iteration count (its tolerance is set so wide that any point
meets it).  Everything else is as in a solve to tolerance: scaling, power
iteration, checks and restarts every 64 iterations, Algorithm 1, reports.

`exact` restates the method with torch in 64 bits, independently of the
library: scaling, both inner loops with their restarts, Algorithm 1 and its
dual counterpart, the KKT numbers, and the guidance network.
"""
import ctypes
import math

import numpy as np
import torch

import lpgen
from paper_2511_13894_gb300 import pdhgc as P

WIDE = 1e30  # a corner tolerance that any point meets


def listed():
    return [
        # the smallest LP, both phases: a service that corners many small LPs one by one; latency decides
        dict(name="face_200x500", kind="solve", lp="face", m=200, n=500, algorithm="halpern", precision="fp64",
             iters=512, corner="primal", corner_iters=2048),
        # the guidance recipe's training size: a small general-form LP with skewed columns, both phases
        dict(name="power_2000x8000", kind="solve", lp="power", m=2000, n=8000, algorithm="halpern",
             precision="fp64", iters=1024, corner="primal", corner_iters=1024),
        # the default inner loop (averaged) on a ragged mid-size LP with '<', '>' rows and boxes, then the
        # dual corner push
        dict(name="bounded_4999x17501_avg", kind="solve", lp="bounded", m=4999, n=17501, algorithm="averaged",
             precision="fp64", iters=1000, corner="dual", corner_iters=512),
        # the guidance recipe's full size, both phases: the ordinary LP
        dict(name="power_20kx80k", kind="solve", lp="power", m=20000, n=80000, algorithm="halpern",
             precision="fp64", iters=1024, corner="primal", corner_iters=1024),
        # the same size in FP32 bulk with the averaged loop
        dict(name="power_20kx80k_avg_fp32", kind="solve", lp="power", m=20000, n=80000, algorithm="averaged",
             precision="fp32", iters=1024, corner="none", corner_iters=0),
        # the benchmark's headline LP, phase 1 in FP64
        dict(name="power_100kx400k", kind="solve", lp="power", m=100000, n=400000, algorithm="halpern",
             precision="fp64", iters=1024, corner="none", corner_iters=0),
        # the headline LP in FP32 bulk
        dict(name="power_100kx400k_fp32", kind="solve", lp="power", m=100000, n=400000, algorithm="halpern",
             precision="fp32", iters=1024, corner="none", corner_iters=0),
        # the transportation workload: two million two-entry columns, long rows, both phases
        dict(name="transport_1000x2000", kind="solve", lp="transport", m=1000, n=2000, algorithm="halpern",
             precision="fp64", iters=256, corner="primal", corner_iters=256),
        # many uneven LPs in one call (the batch recipe), FP32 bulk, both phases fused
        dict(name="batch_192", kind="batch", count=192, mlo=50, mhi=5000, precision="fp32", iters=256,
             corner_iters=256),
        # scoring a point the user holds on the device, without a handle (the headline size)
        dict(name="kkt_eval_100kx400k", kind="kkt", lp="power", m=100000, n=400000),
        # the guidance network: probabilities of an 80k-column LP
        dict(name="guide_infer_80k", kind="infer", rows=80000),
        # the guidance network: minibatch Adam steps on a dataset of 80k rows
        dict(name="guide_train_80k", kind="train", rows=80000, batch=4096, steps=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["batch", "kkt", "infer", "train"])
    if kind == "batch":
        mhi = _log(rng, 500, 5000)
        return dict(kind="batch", count=_log(rng, 24, 192), mlo=50, mhi=mhi,
                    precision=rng.choice(["fp32", "fp64"]), iters=rng.randint(100, 256),
                    corner_iters=64 * rng.randint(2, 4))
    if kind == "kkt":
        m = _log(rng, 1000, 100000)
        return dict(kind="kkt", lp="power", m=m, n=4 * m - rng.randint(0, m // 8))
    if kind == "infer":
        return dict(kind="infer", rows=_log(rng, 500, 80000))
    if kind == "train":
        return dict(kind="train", rows=_log(rng, 5000, 80000), batch=_log(rng, 256, 4096), steps=rng.randint(16, 64))
    lp = rng.choice(["face", "bounded", "power", "power", "transport"])
    if lp == "transport":
        m = _log(rng, 30, 900)
        n = _log(rng, 30, 1900)
    elif lp == "power":
        m = _log(rng, 1000, 90000)
        n = 4 * m - rng.randint(0, m // 8)
    else:
        m = _log(rng, 100, 8000)
        n = int(m * rng.uniform(2.0, 4.0))
    corner = rng.choice(["none", "primal", "primal", "dual"]) if lp == "bounded" else rng.choice(["none", "primal"])
    big = lp == "transport" or m > 30000
    return dict(kind="solve", lp=lp, m=m, n=n, algorithm=rng.choice(["halpern", "halpern", "averaged"]),
                precision=rng.choice(["fp64", "fp64", "fp32"]), iters=rng.randint(100, 256 if big else 1024),
                corner=corner, corner_iters=0 if corner == "none" else 64 * rng.randint(2, 4 if big else 16))


# ---- inputs -----------------------------------------------------------------

def _lp(case, seed):
    m, n = case["m"], case["n"]
    if case["lp"] == "transport":
        return lpgen.transportation_lp(m, n, seed)
    if case["lp"] == "power":
        # the guidance recipes' supports: m + m / 20 columns off their bounds
        return lpgen.power_law_lp(m, n, m // 20, seed, kmax=500 if m <= 5000 else 2000)
    lp = lpgen.random_face_lp(m, n, m + m // 4, seed)
    return lpgen.with_bounds_and_inequalities(lp, seed) if case["lp"] == "bounded" else lp


def _batch(case, seed):
    """The batch recipe: m uniform in its range, n = 2 to 4 times m, 3 to 12 entries a column; the sizes belong
    to the case, the entries to the seed."""
    r = np.random.default_rng(case["count"])
    lps = []
    for i in range(case["count"]):
        m = int(r.integers(case["mlo"], case["mhi"] + 1))
        n = int(round(r.uniform(2.0, 4.0) * m))
        lps.append(lpgen.random_face_lp(m, n, m + math.ceil(m / 4), seed * 1000 + i, col_nnz_range=(3, 12)))
    return lps


def _point(lp, seed):
    """A point near the optimum, as a solver under development hands it over."""
    r = np.random.default_rng(seed)
    return (lp["x_star"] + 1e-2 * r.standard_normal(lp["n"]) * (r.random(lp["n"]) < 0.5),
            lp["y_star"] + 1e-2 * r.standard_normal(lp["m"]))


def _dataset(case, seed):
    """Feature rows (18 used of 32, unit-size groups) and labels of a separable rule with noise."""
    r = np.random.default_rng(seed)
    f = np.zeros((case["rows"], P.GUIDE_FEAT_STRIDE), dtype=np.float32)
    f[:, :18] = r.standard_normal((case["rows"], 18))
    f[:, 1:10] = np.abs(f[:, 1:10])  # column norms and primal histories are nonnegative
    rule = f[:, :18] @ r.standard_normal(18) + 0.5 * r.standard_normal(case["rows"])
    w = np.zeros(P.GUIDE_PARAMS, dtype=np.float32)
    w[:1152] = r.standard_normal(1152) * math.sqrt(2.0 / 18)
    w[1216:5312] = r.standard_normal(4096) * math.sqrt(2.0 / 64)
    w[5376:5440] = r.standard_normal(64) * math.sqrt(1.0 / 64)
    return f, (rule > np.quantile(rule, 0.68)).astype(np.uint8), w


def _params(case, kw=None):
    return dict(algorithm=P.HALPERN if case.get("algorithm", "halpern") == "halpern" else P.AVERAGED,
                precision=P.FP64 if case["precision"] == "fp64" else P.FP32_BULK, eps_rel=-1.0,
                max_iters=case["iters"])


def _corner_params(case):
    return dict(obj_seed=7, eps_rel=WIDE, min_iters=case["corner_iters"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return dict(case=case, lp=P.lp_from_dict(_lp(case, seed)))
    if kind == "batch":
        return dict(case=case, batch=P.Batch(_batch(case, seed)))
    if kind == "kkt":
        lp = _lp(case, seed)
        x, y = _point(lp, seed)
        dev = {k: torch.as_tensor(lp[k]).cuda() for k in ("row_ptr", "col_idx", "val", "b", "c", "lb", "ub", "sense")}
        dev.update(x=torch.as_tensor(x).cuda(), y=torch.as_tensor(y).cuda())
        return dict(case=case, m=lp["m"], n=lp["n"], nnz=int(lp["row_ptr"][-1]), dev=dev)
    f, labels, w = _dataset(case, seed)
    net = P.Guide(seed=0)
    net.set_weights(w)
    return dict(case=case, net=net, w=w, feat=torch.as_tensor(f).cuda().to(torch.bfloat16),
                labels=torch.as_tensor(labels).cuda(), seed=seed)


# ---- one pass ---------------------------------------------------------------

def _counts(r):
    return [r["status"], r["iters"], r["restarts"], r["off_bound_p"], r["zero_rc_d"], r["candidates"]]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        g = state["lp"]
        r = g.solve(**_params(case))
        out = dict(counts=_counts(r), pobj=r["pobj"], dobj=r["dobj"])
        out["x"], out["y"], out["z"] = g.get_solution(P.PHASE1, device=True)
        if case["corner"] == "primal":
            r = g.corner_phase(**_corner_params(case))
            out["corner_x"], _, _ = g.get_solution(P.CORNER, device=True)
        elif case["corner"] == "dual":
            r = g.dual_corner_phase(**_corner_params(case))
            _, out["corner_y"], out["corner_z"] = g.get_solution(P.DUAL_CORNER, device=True)
        if case["corner"] != "none":
            out["corner_counts"] = _counts(r)
        it = g.get_iterates(device=True)
        out["it"] = [it["x"], it["y"], it["x_avg"], it["y_avg"]]
        return out
    if kind == "batch":
        b = state["batch"]
        r1, rc = b.solve_corner(P.default_params(**_params(case)), P.default_corner_params(**_corner_params(case)))
        one = [b.get_solution(k, P.PHASE1) for k in range(b.count)]
        two = [b.get_solution(k, P.CORNER) for k in range(b.count)]
        return dict(x=np.concatenate([v[0] for v in one]), y=np.concatenate([v[1] for v in one]),
                    corner_x=np.concatenate([v[0] for v in two]),
                    counts=np.array([_counts(r) for r in r1]), corner_counts=np.array([_counts(r) for r in rc]))
    if kind == "kkt":
        r = P.Report()
        d = {k: v.data_ptr() for k, v in state["dev"].items()}
        rc = P.lib.pdhgc_kkt_eval(state["m"], state["n"], state["nnz"], d["row_ptr"], d["col_idx"], d["val"], d["b"],
                                  d["c"], d["lb"], d["ub"], d["sense"], d["x"], d["y"], ctypes.byref(r),
                                  torch.cuda.current_stream().cuda_stream)
        if rc != P.OK:
            raise P.PdhgcError(rc, "pdhgc_kkt_eval")
        return dict(kkt=np.array([r.rP2, r.rD2, r.rPinf, r.rDinf, r.pobj, r.dobj, r.gap, r.rel_p, r.rel_d,
                                  r.rel_gap]), counts=[r.off_bound_p, r.zero_rc_d, r.candidates])
    if kind == "infer":
        return state["net"].infer(state["feat"])
    # a training run starts from the user's weights
    net = state["net"]
    net.set_weights(state["w"])
    losses = net.train(state["feat"], state["labels"], rows=case["rows"], batch=case["batch"], steps=case["steps"],
                       lr=1e-3, seed=state["seed"])
    return dict(losses=losses, weights=net.get_weights())


def _nnz(case):
    if case["lp"] == "transport":
        return 2 * case["m"] * case["n"], case["m"] + case["n"], case["m"] * case["n"]
    return (8 if case["lp"] == "power" else 5) * case["n"], case["m"], case["n"]


def work(case):
    """Bytes: the matrix (values and indices, once), the vectors and the results.  Flops: the products of
    A and A' and the vector updates of every iteration."""
    kind = case["kind"]
    if kind in ("solve", "kkt"):
        nnz, m, n = _nnz(case)
        bytes_ = 12 * nnz + 8 * (5 * n + 3 * m)
        if kind == "kkt":
            return dict(bytes=bytes_, flops=4 * nnz + 12 * n + 8 * m)
        its = case["iters"] + case["corner_iters"]
        return dict(bytes=bytes_, flops=its * (4.0 * nnz + 10 * n + 10 * m))
    if kind == "batch":
        m = 0.5 * (case["mlo"] + case["mhi"]) * case["count"]
        n, nnz = 3 * m, 22.5 * m
        its = case["iters"] + case["corner_iters"]
        return dict(bytes=12 * nnz + 8 * (5 * n + 3 * m), flops=its * (4.0 * nnz + 10 * n + 10 * m))
    per_row = 2.0 * (18 * 64 + 64 * 64 + 64)
    if kind == "infer":
        return dict(bytes=case["rows"] * 68, flops=case["rows"] * per_row)
    return dict(bytes=case["steps"] * case["batch"] * 65, flops=3 * case["steps"] * case["batch"] * per_row)


# ---- the same results in 64 bits --------------------------------------------

def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _mix(seed, count, first=0):
    """Outputs first + 1 .. first + count of SplitMix64 (Steele, Lea and Flood 2014) started at `seed`."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(first + 1, first + count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _uniform(seed, count):
    return (_mix(seed, count) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


class _Exact:
    """The method on one LP, or on several side by side (a block-diagonal matrix whose blocks have their own
    step sizes, weights and restarts)."""

    def __init__(self, lps):
        f = lambda key: torch.as_tensor(np.concatenate([lp[key] for lp in lps])).to(_dev())  # noqa: E731
        self.L = len(lps)
        self.ms, self.ns = [lp["m"] for lp in lps], [lp["n"] for lp in lps]
        self.m, self.n = sum(self.ms), sum(self.ns)
        seg = lambda sizes: torch.as_tensor(np.repeat(np.arange(self.L), sizes)).to(_dev())  # noqa: E731
        self.rseg, self.cseg = seg(self.ms), seg(self.ns)
        row = np.concatenate([np.repeat(np.arange(lp["m"]), np.diff(lp["row_ptr"])) + o
                              for lp, o in zip(lps, np.cumsum([0] + self.ms))])
        col = np.concatenate([lp["col_idx"].astype(np.int64) + o for lp, o in zip(lps, np.cumsum([0] + self.ns))])
        self.row, self.col = torch.as_tensor(row).to(_dev()), torch.as_tensor(col).to(_dev())
        sense = f("sense")
        self.sign = torch.where(sense == lpgen.LE, -1.0, 1.0).double()
        self.ge = sense != lpgen.EQ
        self.val = f("val") * self.sign[self.row]
        self.b_user, self.c_user, self.l, self.u = f("b"), f("c"), f("lb"), f("ub")
        self.zero = torch.zeros_like(self.ge)  # rows whose dual is fixed at 0
        # ten Ruiz passes, then Pock-Chambolle
        dr, dc = torch.ones(self.m).double().to(_dev()), torch.ones(self.n).double().to(_dev())
        a = self.val.abs()
        fac = lambda v: torch.where(v > 0, 1.0 / torch.sqrt(torch.where(v > 0, v, 1.0)), 1.0)  # noqa: E731
        for _ in range(10):
            e = dr[self.row] * a * dc[self.col]
            r = torch.zeros_like(dr).scatter_reduce(0, self.row, e, "amax")
            c = torch.zeros_like(dc).scatter_reduce(0, self.col, e, "amax")
            dr, dc = dr * fac(r), dc * fac(c)
        e = dr[self.row] * a * dc[self.col]
        r = torch.zeros_like(dr).index_add(0, self.row, e)
        c = torch.zeros_like(dc).index_add(0, self.col, e)
        self.dr, self.dc = dr * fac(r), dc * fac(c)
        hat = self.dr[self.row] * self.val * self.dc[self.col]

        def csr(i, j, shape):
            order = torch.argsort(i, stable=True)
            ptr = torch.zeros(shape[0] + 1, dtype=torch.int64, device=_dev())
            ptr[1:] = torch.cumsum(torch.bincount(i, minlength=shape[0]), 0)
            return torch.sparse_csr_tensor(ptr, j[order], hat[order], shape)
        self.A, self.T = csr(self.row, self.col, (self.m, self.n)), csr(self.col, self.row, (self.n, self.m))
        self.b, self.c = self.dr * self.sign * self.b_user, self.dc * self.c_user
        self.lh, self.uh = self.l / self.dc, self.u / self.dc
        self.nb, self.nc = self._norm(self.b_user, 0), self._norm(self.c_user, 1)
        v = torch.as_tensor(np.repeat(1.0 / np.sqrt(np.array(self.ns, dtype=np.float64)), self.ns)).to(_dev())
        for _ in range(100):
            w = self.T @ (self.A @ v)
            v = w / self._of(self._norm(w, 1), 1)
        self.eta = 0.998 / self._norm(self.A @ v, 0)

    def _sum(self, v, side):
        """Sums per LP (side 0: rows, 1: columns), as a numpy array."""
        if self.L == 1:
            return v.sum().reshape(1).cpu().numpy()
        seg = self.cseg if side else self.rseg
        return torch.zeros(self.L, dtype=torch.float64, device=_dev()).index_add(0, seg, v).cpu().numpy()

    def _norm(self, v, side):
        return np.sqrt(self._sum(v * v, side))

    def _of(self, a, side):
        """The LPs' own values as one per row (side 0) or column (1)."""
        t = torch.as_tensor(np.asarray(a, dtype=np.float64)).to(_dev())
        return t if self.L == 1 else t[self.cseg if side else self.rseg]

    def reduced(self, lam):
        lf, uf = torch.isfinite(self.lh), torch.isfinite(self.uh)
        z = torch.where(uf, lam.clamp(max=0.0), torch.zeros_like(lam))
        return torch.where(lf, torch.where(uf, lam, lam.clamp(min=0.0)), z)

    def _kkt(self, x, y):
        """Squared scaled residuals, the gap and both objectives, per LP."""
        r = self.b - self.A @ x
        r = torch.where(self.zero, 0.0, torch.where(self.ge, r.clamp(min=0.0), r))
        lam = self.c - self.T @ y
        z = self.reduced(lam)
        bound = (torch.where(torch.isfinite(self.lh), self.lh, 0.0) * z.clamp(min=0.0)
                 - torch.where(torch.isfinite(self.uh), self.uh, 0.0) * (-z).clamp(min=0.0))
        pobj = self._sum(self.c * x, 1)
        dobj = self._sum(self.b * y, 0) + self._sum(bound, 1)
        rd = lam - z
        nc = self._norm(self.c / self.dc, 1)
        rel = np.maximum(self._norm(r / self.dr, 0) / (1 + self.nb), self._norm(rd / self.dc, 1) / (1 + nc))
        rel = np.maximum(rel, np.abs(pobj - dobj) / (1 + np.abs(pobj) + np.abs(dobj)))
        return dict(p=self._sum(r * r, 0), d=self._sum(rd * rd, 1), gap=pobj - dobj, pobj=pobj, dobj=dobj, rel=rel)

    def phase(self, iters, halpern, x, y, corner=False):
        """`iters` iterations from (x, y) with the checks, restarts and weight updates of the loop; returns the
        returned point and the final iterates (current; average, or the operator's output)."""
        L = self.L
        nch, nbh = self._norm(self.c, 1), self._norm(self.b, 0)
        om = np.where((nch > 1e-10) & (nbh > 1e-10), nch / np.where(nbh > 0, nbh, 1.0), 1.0)
        tau, sig = self.eta / om, self.eta * om
        t, k, prev = np.zeros(L), 0, np.full(L, math.inf)
        xr, yr, sx, sy = x, y, torch.zeros_like(x), torch.zeros_like(y)
        integral, eprev = np.zeros(L), np.zeros(L)

        def operator(x, y):
            xp = torch.minimum(torch.maximum(x - self._of(tau, 1) * (self.c - self.T @ y), self.lh), self.uh)
            yp = y + self._of(sig, 0) * (self.b - self.A @ (2.0 * xp - x))
            return xp, torch.where(self.zero, 0.0, torch.where(self.ge, yp.clamp(min=0.0), yp))

        def residual(dx, dy):
            q = self._sum(dx * dx, 1) / tau + self._sum(dy * dy, 0) / sig + 2 * self._sum(dy * (self.A @ dx), 0)
            return np.sqrt(np.maximum(q, 0.0))
        weigh = lambda e, w: np.sqrt(w * e["p"] + e["d"] / w + e["gap"] ** 2)  # noqa: E731
        if halpern:
            xp, yp = operator(x, y)
            ref = residual(x - xp, y - yp)
        else:
            xp, yp, ref = x, y, weigh(self._kkt(x, y), om)
        while True:
            taus, sigs = tau, sig
            for _ in range(min(64, iters - k)):
                x0, y0 = x, y
                xp, yp = operator(x, y)
                if halpern:
                    w = (t + 1) / (t + 2)
                    wx, wy = self._of(w, 1), self._of(w, 0)
                    x = wx * (2.0 * xp - x) + (1.0 - wx) * xr
                    y = wy * (2.0 * yp - y) + (1.0 - wy) * yr
                else:
                    x, y, sx, sy = xp, yp, sx + xp, sy + yp
                t, k = t + 1, k + 1
            assert taus is tau and sigs is sig
            if k >= iters:
                break
            if halpern:
                r = residual(x0 - xp, y0 - yp)
                go = (r <= 0.2 * ref) | ((r <= 0.8 * ref) & (r > prev)) | (t >= 0.36 * k)
                dx, dy = self._norm(xp - xr, 1), self._norm(yp - yr, 0)
                for i in np.nonzero(go & (dx > 1e-10) & (dy > 1e-10))[0]:
                    e = math.log(om[i]) - math.log(dy[i] / dx[i])
                    integral[i] += e
                    om[i] = math.exp(math.log(om[i]) - (0.99 * e + 0.01 * integral[i]))
                    eprev[i] = e
                ref, cx, cy = np.where(go, r, ref), xp, yp
            else:
                xa, ya = sx / self._of(t, 1), sy / self._of(t, 0)
                e0, e1 = self._kkt(x, y), self._kkt(xa, ya)
                avg = weigh(e1, om) <= weigh(e0, om)
                ev = {q: np.where(avg, e1[q], e0[q]) for q in e0}
                r = weigh(ev, om)
                go = (r <= 0.2 * ref) | ((r <= 0.8 * ref) & (r > prev)) | (t >= 0.36 * k)
                ax, ay = self._of(avg, 1) > 0, self._of(avg, 0) > 0
                cx, cy = torch.where(ax, xa, x), torch.where(ay, ya, y)
                dx, dy = self._norm(cx - xr, 1), self._norm(cy - yr, 0)
                for i in np.nonzero(go & (dx > 1e-10) & (dy > 1e-10))[0]:
                    om[i] = math.exp(0.5 * math.log(dy[i] / dx[i]) + 0.5 * math.log(om[i]))
                ref = np.where(go, weigh(ev, om), ref)
            prev = np.where(go, math.inf, r)
            gx, gy = self._of(go, 1) > 0, self._of(go, 0) > 0
            x, y = torch.where(gx, cx, x), torch.where(gy, cy, y)
            xr, yr = torch.where(gx, cx, xr), torch.where(gy, cy, yr)
            sx, sy = torch.where(gx, 0.0, sx), torch.where(gy, 0.0, sy)
            t = np.where(go, 0.0, t)
            tau, sig = self.eta / om, self.eta * om
        if halpern:
            return (xp, yp), (x, y, xp, yp)
        xa, ya = sx / self._of(t, 1), sy / self._of(t, 0)
        pick = np.zeros(L, dtype=bool) if corner else self._kkt(xa, ya)["rel"] <= self._kkt(x, y)["rel"]
        ax, ay = self._of(pick, 1) > 0, self._of(pick, 0) > 0
        return (torch.where(ax, xa, x), torch.where(ay, ya, y)), (x, y, xa, ya)

    def phase1(self, iters, halpern):
        zero = torch.zeros_like(self.c)
        return self.phase(iters, halpern, torch.minimum(torch.maximum(zero, self.lh), self.uh),
                          torch.zeros_like(self.b))

    def user(self, x, y):
        return self.dc * x, self.sign * self.dr * y, self.reduced(self.c - self.T @ y) / self.dc

    def corner(self, x1, y1, iters, halpern):
        """Algorithm 1 from the scaled phase-1 point (objective seed 7)."""
        z = self.reduced(self.c - self.T @ y1) / self.dc
        keep = (self.c, self.lh, self.uh, self.ge)
        obj = torch.as_tensor(np.concatenate([_uniform(7, n) for n in self.ns])).to(_dev())
        self.c = self.dc * obj
        self.uh, self.lh = torch.where(z > 1e-6, x1, self.uh), torch.where(z < -1e-6, x1, self.lh)
        self.ge = self.ge & ~((self.dr * y1).abs() > 1e-6)
        got = self.phase(iters, halpern, x1, torch.zeros_like(self.b), corner=True)
        self.c, self.lh, self.uh, self.ge = keep
        return got

    def dual_corner(self, x1, y1, iters, halpern):
        """The dual corner push from the scaled phase-1 point (objective seed 7)."""
        x, _, z = self.user(x1, y1)
        keep = (self.b, self.lh, self.uh, self.zero)
        dl, du = x - self.l, self.u - x
        off_l, off_u = (dl > 1e-6) & (dl > z.clamp(min=0.0)), (du > 1e-6) & (du > (-z).clamp(min=0.0))
        slack = (self.A @ x1) / self.dr - self.sign * self.b_user
        self.zero = self.ge & (slack > 1e-6) & (slack > (self.dr * y1).abs())
        self.lh, self.uh = torch.where(off_l, -math.inf, self.lh), torch.where(off_u, math.inf, self.uh)
        obj = torch.as_tensor(np.concatenate([_uniform(7, m) for m in self.ms])).to(_dev())
        self.b = torch.where(self.zero, 0.0, self.dr * self.sign * obj)
        x0 = torch.minimum(torch.maximum(torch.zeros_like(self.c), self.lh), self.uh)
        got = self.phase(iters, halpern, x0, torch.where(self.zero, 0.0, y1), corner=True)
        self.b, self.lh, self.uh, self.zero = keep
        return got


def _exact_solve(case, seed):
    e = _Exact([_lp(case, seed)])
    halpern = case["algorithm"] == "halpern"
    (x1, y1), its = e.phase1(case["iters"], halpern)
    k = e._kkt(x1, y1)
    out = dict(counts=[None] * 6, pobj=float(k["pobj"][0]), dobj=float(k["dobj"][0]))
    out["x"], out["y"], out["z"] = e.user(x1, y1)
    if case["corner"] == "primal":
        (xc, _), its = e.corner(x1, y1, case["corner_iters"], halpern)
        out["corner_x"] = e.dc * xc
    elif case["corner"] == "dual":
        (_, yd), its = e.dual_corner(x1, y1, case["corner_iters"], halpern)
        _, out["corner_y"], out["corner_z"] = e.user(x1, yd)
    out["it"] = list(its)
    return out


def _exact_batch(case, seed):
    e = _Exact(_batch(case, seed))
    (x1, y1), _ = e.phase1(case["iters"], True)
    (xc, _), _ = e.corner(x1, y1, case["corner_iters"], True)
    x, y, _ = e.user(x1, y1)
    return dict(x=x, y=y, corner_x=e.dc * xc, counts=None, corner_counts=None)


def _exact_kkt(case, seed):
    lp = _lp(case, seed)
    x, y = _point(lp, seed)
    row = np.repeat(np.arange(lp["m"]), np.diff(lp["row_ptr"]))
    ax = np.bincount(row, lp["val"] * x[lp["col_idx"]], lp["m"])
    lam = lp["c"] - np.bincount(lp["col_idx"], lp["val"] * y[row], lp["n"])
    r = lp["b"] - ax
    r = np.where(lp["sense"] == lpgen.LE, np.minimum(r, 0.0), r)
    r = np.where(lp["sense"] == lpgen.GE, np.maximum(r, 0.0), r)
    lf, uf = np.isfinite(lp["lb"]), np.isfinite(lp["ub"])
    z = np.where(lf & uf, lam, np.where(lf, np.maximum(lam, 0.0), np.where(uf, np.minimum(lam, 0.0), 0.0)))
    rd = lam - z
    pobj = lp["c"] @ x
    dobj = lp["b"] @ y + (np.where(lf, lp["lb"], 0) @ np.maximum(z, 0)) - (np.where(uf, lp["ub"], 0) @ np.maximum(-z, 0))
    n = np.linalg.norm
    return dict(kkt=np.array([n(r), n(rd), np.abs(r).max(), np.abs(rd).max(), pobj, dobj, pobj - dobj,
                              n(r) / (1 + n(lp["b"])), n(rd) / (1 + n(lp["c"])),
                              abs(pobj - dobj) / (1 + abs(pobj) + abs(dobj))]), counts=[None] * 3)


def _unpack(w):
    w = torch.as_tensor(w).double().to(_dev())
    return [w[:1152].reshape(64, 18), w[1152:1216], w[1216:5312].reshape(64, 64), w[5312:5376], w[5376:5440], w[5440:]]


def _logits(w, x):
    h = torch.relu(x @ w[0].T + w[1])
    return torch.relu(h @ w[2].T + w[3]) @ w[4] + w[5]


def _exact_net(case, seed):
    f, labels, w = _dataset(case, seed)
    x = torch.as_tensor(f).to(torch.bfloat16).double().to(_dev())[:, :18]
    w = [v.requires_grad_(case["kind"] == "train") for v in _unpack(w)]
    if case["kind"] == "infer":
        return torch.sigmoid(_logits(w, x))
    y = torch.as_tensor(labels).double().to(_dev())
    opt = torch.optim.Adam(w, lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
    losses = []
    for s in range(case["steps"]):
        rows = torch.as_tensor((_mix(seed, case["batch"], s * case["batch"]) % np.uint64(case["rows"])).astype(np.int64))
        rows = rows.to(_dev())
        loss = torch.nn.functional.binary_cross_entropy_with_logits(_logits(w, x[rows]), y[rows])
        opt.zero_grad()
        loss.backward()
        opt.step()
        losses.append(loss.detach())
    return dict(losses=torch.stack(losses), weights=torch.cat([v.detach().reshape(-1) for v in w]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return _exact_solve(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    return _exact_kkt(case, seed) if kind == "kkt" else _exact_net(case, seed)
