"""The work that users of this library have it do, as measurable cases.

A case is one call sequence through the public Python binding, at a stated
size.  Kinds:

* center    pdhg.centered_point_noalloc: the start point of caller's vectors;
* oneshot   an LP handed over once: create, solve to 1e-4, solution and start
            point, destroy;
* solve     a kept solver: from the stored state to 1e-4, then the solution;
* iterate   a kept solver: a fixed number of iterations from a stored state,
            then the solver's state (checkpointed running);
* create    the set-up of a solver alone: transpose, scaling, step size, tuning;
* finish    the solution, its residuals and the start point of an iterate;
* batch     a kept batch of LPs with new right-hand sides: solve, solutions;
* autograd  forward and backward of x*(b, c) for a batch of LPs with fixed A.

LP families: planted (5 nonzeros per column), powerlaw (heavy-tailed row
lengths, 1% of the rows scaled by 1e3), transport (balanced transportation).
In float32-mixed solvers every iterate is a float32 number; the state calls
widen it, and these cases hand it on as the float32 numbers it is (exact for
a solver's state; a batch's solution is the float32 iterate times its float64
scaling, rounded once).
"""
import math

import numpy as np
import torch

from paper_2603_03150_gb300 import autograd, pdhg

EPS = 1e-4         # the hand-over tolerance of every solve
MAX_ITER = 200_000


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # an interior-point code asking for the start point of a small LP's
        # vectors inside its own loop: launches and latency only
        dict(name="center_500", kind="center", n=500),
        # the small configuration (200 x 500), handed over once, default options
        dict(name="oneshot_200x500", kind="oneshot", family="planted", m=200, n=500, precision="fp64"),
        # a service that keeps solvers of ordinary LPs (2000 x 5000): latency per iteration
        dict(name="solve_2000x5000", kind="solve", family="planted", m=2000, n=5000, precision="fp64"),
        # the main workload: 200k x 1M, 5M nonzeros, float32-mixed, averaged method
        dict(name="iterate_powerlaw_fp32", kind="iterate", family="powerlaw", m=200_000, n=1_000_000,
             nnz=5_000_000, precision="fp32", iters=128, rule="averaged"),
        # the same LP in float64, the default precision
        dict(name="iterate_powerlaw_fp64", kind="iterate", family="powerlaw", m=200_000, n=1_000_000,
             nnz=5_000_000, precision="fp64", iters=64, rule="averaged"),
        # the large transportation LP, reflected Halpern iteration with PID weight
        dict(name="iterate_transport_halpern", kind="iterate", family="transport", m=2000, n=2000,
             precision="fp32", iters=64, rule="halpern_pid"),
        # a ragged mid-size transportation LP with the adaptive step, float64
        dict(name="iterate_transport_adaptive", kind="iterate", family="transport", m=301, n=707,
             precision="fp64", iters=48, rule="adaptive"),
        # set-up of the main workload (paid once per LP)
        dict(name="create_powerlaw", kind="create", family="powerlaw", m=200_000, n=1_000_000,
             nnz=5_000_000, precision="fp32"),
        # what follows a solve of the main workload: solution, residuals, start point
        dict(name="finish_powerlaw", kind="finish", family="powerlaw", m=200_000, n=1_000_000,
             nnz=5_000_000, precision="fp32"),
        # 512 uneven LPs (m log-uniform in 50..5000) solved together, float64
        dict(name="batch_512_fp64", kind="batch", count=512, m_lo=50, m_hi=5000, precision="fp64",
             iters=0),
        # an uneven, smaller batch in float32-mixed, a fixed number of iterations
        dict(name="batch_97_fp32", kind="batch", count=97, m_lo=50, m_hi=5000, precision="fp32",
             iters=192),
        # differentiation: 64 LPs of 2000 x 5000, forward and backward
        dict(name="autograd_64", kind="autograd", count=64, m=2000, n=5000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["center", "oneshot", "solve", "iterate", "iterate", "iterate", "create",
                       "finish", "batch", "batch", "autograd"])
    prec = rng.choice(["fp64", "fp32"])
    if kind == "center":
        return dict(kind=kind, n=_log_int(rng, 20, 8_000_000))
    if kind in ("oneshot", "solve"):
        m = _log_int(rng, 100, 6000)
        return dict(kind=kind, family="planted", m=m, n=int(m * rng.uniform(2.2, 3.0)), precision="fp64")
    if kind in ("iterate", "create", "finish"):
        family = rng.choice(["planted", "powerlaw", "transport"])
        case = dict(kind=kind, family=family, precision=prec)
        if family == "transport":
            case.update(m=_log_int(rng, 30, 2000), n=_log_int(rng, 30, 2000))
        elif family == "planted":
            m = _log_int(rng, 150, 100_000)
            case.update(m=m, n=int(m * rng.uniform(2.2, 3.0)))
        else:
            m = _log_int(rng, 2000, 200_000)
            case.update(m=m, n=int(4.7 * m), nnz=25 * m)
        if kind == "iterate":
            # the adaptive step carries every rounding into the next step, so
            # it is drawn in float64 and for fewer steps
            rules = ["averaged", "halpern", "averaged_pid", "halpern_pid"]
            case.update(iters=rng.randrange(33, 129), rule=rng.choice(rules + ["adaptive"] * (prec == "fp64")))
            if case["rule"] == "adaptive":
                case["iters"] = rng.randrange(17, 49)
        return case
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 3, 500), m_lo=50, m_hi=_log_int(rng, 100, 5000),
                    precision=prec, iters=0 if prec == "fp64" else rng.randrange(65, 193))
    m = _log_int(rng, 100, 2000)
    return dict(kind=kind, count=_log_int(rng, 2, 64), m=m, n=int(2.5 * m))


# ---------------------------------------------------------------------------
# inputs (made on the GPU from the seed alone)
# ---------------------------------------------------------------------------
def _segment_sum(v, lengths):
    """Sums of consecutive segments of v (a fixed order)."""
    return torch.segment_reduce(v, "sum", lengths=lengths, initial=0.0)


class _LP:
    """A block-diagonal stack of LPs (one for a single LP), columns global."""

    def __init__(self, ms, ns, key, val):
        # key = row * N + column, distinct, in any order
        dev = key.device
        self.ms, self.ns = np.asarray(ms, np.int64), np.asarray(ns, np.int64)
        self.m, self.n = int(self.ms.sum()), int(self.ns.sum())
        key, order = torch.sort(key)
        self.row, self.col, self.val = key // self.n, key % self.n, val[order]
        self.row_len = torch.bincount(self.row, minlength=self.m)
        self.lp_of_row = torch.repeat_interleave(torch.arange(len(ms), device=dev),
                                                 torch.as_tensor(self.ms, device=dev))
        self.lp_of_col = torch.repeat_interleave(torch.arange(len(ns), device=dev),
                                                 torch.as_tensor(self.ns, device=dev))

    def times(self, v):
        return _segment_sum(self.val * v[self.col], self.row_len)

    def transposed_times(self, u):
        _, order = torch.sort(self.col * self.m + self.row)
        return _segment_sum((self.val * u[self.row])[order], torch.bincount(self.col, minlength=self.n))

    def arrays(self):
        """The arrays of the C ABI: per-LP row pointers and local columns."""
        ptr = torch.cat([self.row_len.new_zeros(1), torch.cumsum(self.row_len, 0)])
        if len(self.ms) == 1:
            row_ptr, col = ptr, self.col
        else:
            m_off = np.concatenate([[0], np.cumsum(self.ms)])
            h = ptr.cpu().numpy()
            row_ptr = torch.from_numpy(np.concatenate(
                [h[m_off[i]:m_off[i + 1] + 1] - h[m_off[i]] for i in range(len(self.ms))])).to(ptr.device)
            first = torch.as_tensor(np.concatenate([[0], np.cumsum(self.ns)[:-1]]), device=ptr.device)
            col = self.col - first[self.lp_of_row[self.row]]
        return dict(m=self.ms.astype(np.int32), n=self.ns.astype(np.int32),
                    row_ptr=row_ptr.to(torch.int32).contiguous(), col=col.to(torch.int32).contiguous(),
                    val=self.val.contiguous(), b=self.b.contiguous(), c=self.c.contiguous())


def _plant(lp, gen):
    """b and c with a known optimum: x* > 0 on 30% of the columns, z* > 0 on the rest."""
    dev = lp.val.device
    rand = lambda k: torch.rand(k, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    pos = rand(lp.n) < 0.3
    x = torch.where(pos, 0.5 + 1.5 * rand(lp.n), 0.0)
    z = torch.where(pos, 0.0, 0.5 + 1.5 * rand(lp.n))
    y = torch.randn(lp.m, generator=gen, device=dev, dtype=torch.float64)
    lp.b, lp.c = lp.times(x), lp.transposed_times(y) + z


def _planted(ms, ns, gen, dev):
    """Each column has 5 entries at distinct uniform rows of its LP, values N(0, 1)."""
    ms_t, ns_t = torch.as_tensor(np.asarray(ms), device=dev), torch.as_tensor(np.asarray(ns), device=dev)
    n = int(np.sum(ns))
    lp_of = torch.repeat_interleave(torch.arange(len(ms), device=dev), ns_t)
    rows_of, first = ms_t[lp_of][:, None], (torch.cumsum(ms_t, 0) - ms_t)[lp_of][:, None]

    def draws():
        u = torch.rand((n, 5), generator=gen, device=dev, dtype=torch.float64)
        return torch.minimum((u * rows_of).to(torch.int64), rows_of - 1)

    r = draws()
    while True:
        r = torch.sort(r, 1).values
        again = torch.zeros_like(r, dtype=torch.bool)
        again[:, 1:] = r[:, 1:] == r[:, :-1]
        if not bool(again.any()):
            break
        r = torch.where(again, draws(), r)
    key = ((r + first) * n + torch.arange(n, device=dev)[:, None]).reshape(-1)
    val = torch.randn(5 * n, generator=gen, device=dev, dtype=torch.float64)
    lp = _LP(ms, ns, key, val)
    _plant(lp, gen)
    return lp


def _powerlaw(m, n, nnz, gen, dev):
    """Row lengths P(k) ~ k^-2.1 on [4, 20000], entries added at random rows up
    to about nnz, uniform columns, at least one entry in every column, 1% of
    the rows times 1e3."""
    k_max = min(20_000, n // 4)
    k = torch.arange(4, k_max + 1, device=dev, dtype=torch.float64)
    cdf = torch.cumsum(k.pow(-2.1).cpu(), 0).to(dev)
    u = torch.rand(m, generator=gen, device=dev, dtype=torch.float64) * cdf[-1]
    lens = 4 + torch.searchsorted(cdf, u)
    lens[0] = k_max
    short = nnz - int(lens.sum())
    if short > 0:
        lens += torch.bincount(torch.randint(0, m, (short,), generator=gen, device=dev), minlength=m)
    row = torch.repeat_interleave(torch.arange(m, device=dev), lens)
    col = torch.randint(0, n, (row.numel(),), generator=gen, device=dev)
    bare = torch.nonzero(torch.bincount(col, minlength=n) == 0)[:, 0]
    own = torch.randint(0, m, (bare.numel(),), generator=gen, device=dev)
    key = torch.unique(torch.cat([row * n + col, own * n + bare]))
    scale = torch.where(torch.rand(m, generator=gen, device=dev, dtype=torch.float64) < 0.01, 1e3, 1.0)
    val = torch.randn(key.numel(), generator=gen, device=dev, dtype=torch.float64) * scale[key // n]
    lp = _LP([m], [n], key, val)
    _plant(lp, gen)
    return lp


def _transport(sources, sinks, gen, dev):
    """Arc (i, j) is column i * sinks + j with a 1 in supply row i and demand row j."""
    n = sources * sinks
    arc = torch.arange(n, device=dev)
    key = torch.cat([(arc // sinks) * n + arc, (sources + arc % sinks) * n + arc])
    lp = _LP([sources + sinks], [n], key, torch.ones(2 * n, device=dev, dtype=torch.float64))
    unif = lambda k: 1 + 99 * torch.rand(k, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    s, d = unif(sources).cpu(), unif(sinks).cpu()
    lp.b = torch.cat([s, d * (s.sum() / d.sum())]).to(dev)
    lp.c = unif(n)
    return lp


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(1_000_003 * seed + 17)
    if case["kind"] == "batch":
        rng = np.random.default_rng(case["count"])  # the sizes belong to the case, not to the seed
        ms = np.floor(np.exp(rng.uniform(np.log(case["m_lo"]), np.log(case["m_hi"]), case["count"])))
        ms = ms.astype(np.int64)
        lp = _planted(ms, (5 * ms) // 2, gen, dev)
    elif case["kind"] == "autograd":
        lp = _planted([case["m"]] * case["count"], [case["n"]] * case["count"], gen, dev)
    elif case["family"] == "planted":
        lp = _planted([case["m"]], [case["n"]], gen, dev)
    elif case["family"] == "powerlaw":
        lp = _powerlaw(case["m"], case["n"], case["nnz"], gen, dev)
    else:
        lp = _transport(case["m"], case["n"], gen, dev)
    return lp, gen


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _options(case):
    rule = case.get("rule", "averaged")
    return dict(precision=case["precision"], device_io=True,
                method="halpern" if rule.startswith("halpern") else "averaged",
                omega_rule="pid" if rule.endswith("pid") else "smooth",
                step_rule="adaptive" if rule == "adaptive" else "constant")


def _solver(case, a):
    return pdhg.Solver(a["m"][0], a["n"][0], a["row_ptr"], a["col"], a["val"], a["b"], a["c"],
                       **_options(case))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "center":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(1_000_003 * seed + 17)
        rand = lambda: torch.rand(case["n"], generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
        # complementary pairs: either entry of a pair is near zero
        on = rand() < 0.3
        x, z = torch.where(on, 2 * rand(), 1e-7 * rand()), torch.where(on, 1e-7 * rand(), 2 * rand())
        out = [torch.empty_like(x), torch.empty_like(x), torch.empty(1, device="cuda", dtype=torch.float64)]
        torch.cuda.synchronize()
        return dict(case=case, x=x, z=z, out=out)
    lp, gen = _inputs(case, seed)
    st = dict(case=case, a=lp.arrays())
    if kind == "autograd":
        st["b"], st["c"] = st["a"]["b"].clone().requires_grad_(True), st["a"]["c"]
        st["g"] = torch.randn(lp.n, generator=gen, device="cuda", dtype=torch.float64)
        torch.cuda.synchronize()
        st["lp"] = autograd.BatchLP(st["a"], device="cuda")
        # builds the plan (scaling, transpose, schedules) that the program keeps
        autograd.lp_solution(st["b"].detach(), st["c"], st["lp"], max_iter=0, cg_max_iter=0)
        return st
    torch.cuda.synchronize()  # the library reads the arrays on its own stream
    if kind == "batch":
        st["solver"] = pdhg.BatchSolver(arrays=st["a"], precision=case["precision"], device_io=True)
    elif kind in ("solve", "iterate", "finish"):
        st["solver"] = _solver(case, st["a"])
        if kind == "finish":
            st["solver"].solve(0.0, 64)
        else:
            st["start"] = st["solver"].state()
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "center":
        pdhg.centered_point_noalloc(st["x"], st["z"], *st["out"])
        return st["out"]
    if kind == "autograd":
        x = autograd.lp_solution(st["b"], st["c"], st["lp"], eps_rel=EPS)
        (grad_b,) = torch.autograd.grad(x, st["b"], st["g"])
        return dict(x=x.detach(), grad_b=grad_b)
    if kind == "batch":
        s = st["solver"]
        s.set_rhs(st["a"]["b"], st["a"]["c"])
        s.solve(*((0.0, case["iters"]) if case["iters"] else (EPS, MAX_ITER)))
        g = s.get()
        if case["precision"] == "fp32":
            return dict(x=g["x"].float(), y=g["y"].float(), iters=g["iters"])
        return dict(x=g["x"], y=g["y"], z=g["z"], iters=g["iters"])
    if kind == "create":
        with _solver(case, st["a"]) as s:
            d = s.scaling()
        return dict(D_r=d["D_r"], D_c=d["D_c"], sigma_max=d["sigma_max"], omega0=d["omega0"])
    if kind == "oneshot":
        with _solver(case, st["a"]) as s:
            s.solve(EPS, MAX_ITER)
            return _solution(s, True)
    s = st["solver"]
    if kind == "finish":
        return _solution(s, True)
    s.set_state(st["start"])
    if kind == "solve":
        s.solve(EPS, MAX_ITER)
        return dict(_solution(s, False), iters=s.info(violation=False)["iters"])
    s.solve(0.0, case["iters"])
    d = s.state()
    keep = ("x", "y", "x_avg", "y_avg", "x_last", "y_last", "Ax")
    if case["precision"] == "fp32":
        return {k: d[k].float() for k in keep}  # exact: the iterates are float32 numbers
    return {k: d[k] for k in keep}


def _solution(s, start_point):
    g = s.get()
    out = dict(x=g["x"], y=g["y"], z=g["z"])
    if start_point:
        xw, yw, zw, mu = s.warmstart_point()
        out.update(x_ws=xw, y_ws=yw, z_ws=zw, mu=mu)
    return out


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------
L2_BYTES = 129e6
TYPICAL_ITERS = 640  # iterations to 1e-4 of the planted LPs (about 500 to 1000)
POWER_ITERS = 200
CG_STEPS = 60


def _sizes(case):
    """(m, n, nnz) in total."""
    if case["kind"] == "batch":
        m = case["count"] * (case["m_hi"] - case["m_lo"]) / max(math.log(case["m_hi"] / case["m_lo"]), 1e-9)
        return m, 2.5 * m, 12.5 * m
    if case["kind"] == "autograd":
        return case["count"] * case["m"], case["count"] * case["n"], 5 * case["count"] * case["n"]
    if case["family"] == "transport":
        return case["m"] + case["n"], case["m"] * case["n"], 2 * case["m"] * case["n"]
    return case["m"], case["n"], case["nnz"] if case["family"] == "powerlaw" else 5 * case["n"]


def work(case):
    """Bytes: the inputs and outputs once; where an LP's two matrices do not
    stay in the L2, the matrices, the gathered vectors and the row operands again in
    every iteration.  Flops: a multiply and an add per nonzero and product, and
    the steps' own arithmetic."""
    if case["kind"] == "center":
        return {"bytes": 32.0 * case["n"], "flops": 10.0 * case["n"]}
    m, n, nnz = _sizes(case)
    s = 4.0 if case.get("precision") == "fp32" else 8.0
    lp_bytes = 12.0 * nnz + 4.0 * m + 8.0 * (m + n)
    product = nnz * (4 + s) + 4.0 * (m + n) + s * (m + n)  # one product with A or its transpose
    step = 2 * nnz * (4 + s) + 4.0 * (m + n) + s * (10 * m + 6 * n)
    step_flops = 4.0 * nnz + 12.0 * m + 8.0 * n
    power, power_flops = 2 * (nnz * 12 + 8.0 * (m + n)), 4.0 * nnz + 5.0 * n
    kind = case["kind"]
    # the LPs of a batch are independent: each one alone stays on the chip
    resident = 2 * nnz * (4 + s) < L2_BYTES or kind in ("batch", "autograd")
    its = case.get("iters") or TYPICAL_ITERS
    if kind == "finish":
        return {"bytes": 3 * (12.0 * nnz + 8.0 * (m + n)) + 8.0 * (2 * m + 4 * n), "flops": 6.0 * nnz}
    if kind == "create":
        return {"bytes": lp_bytes + (0 if 24 * nnz < L2_BYTES else POWER_ITERS * power) + product,
                "flops": POWER_ITERS * power_flops + 22 * 4.0 * nnz}
    bytes_, flops = lp_bytes + 8.0 * (m + 2 * n), its * step_flops
    if not resident:
        bytes_ += its * step
    if kind == "oneshot":
        flops += POWER_ITERS * power_flops
    if kind == "autograd":
        flops += 2 * CG_STEPS * (4.0 * nnz + 8.0 * n)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits with plain torch
# ---------------------------------------------------------------------------
class _Plain:
    """Scaled model, step size and the iteration for a stack of LPs."""

    def __init__(self, lp):
        self.lp = lp
        self.k = len(lp.ms)
        self.mlen, self.nlen = (torch.as_tensor(v, device=lp.val.device) for v in (lp.ms, lp.ns))
        t = torch.sort(lp.col * lp.m + lp.row).indices
        self.a_ptr = torch.cat([lp.row_len.new_zeros(1), torch.cumsum(lp.row_len, 0)])
        col_len = torch.bincount(lp.col, minlength=lp.n)
        self.t_ptr = torch.cat([col_len.new_zeros(1), torch.cumsum(col_len, 0)])
        self.t_order, self.t_col = t, lp.row[t]
        d_r, d_c = torch.ones_like(lp.b), torch.ones_like(lp.c)
        for it in range(11):
            v = lp.val.abs() * d_r[lp.row] * d_c[lp.col]
            if it < 10:
                r = torch.zeros_like(d_r).scatter_reduce_(0, lp.row, v, "amax")
                s = torch.zeros_like(d_c).scatter_reduce_(0, lp.col, v, "amax")
            else:
                r = torch.zeros_like(d_r).index_add_(0, lp.row, v)
                s = torch.zeros_like(d_c).index_add_(0, lp.col, v)
            d_r, d_c = (d / torch.where(q == 0, 1.0, q.sqrt()) for d, q in ((d_r, r), (d_c, s)))
        self.d_r, self.d_c = d_r, d_c
        self.set_values(lp.val * d_r[lp.row] * d_c[lp.col])
        self.b, self.c = lp.b * d_r, lp.c * d_c
        self.sigma = self._power()
        self.eta = 0.95 / self.sigma
        nb, nc = self.m_sum(self.b * self.b).sqrt(), self.n_sum(self.c * self.c).sqrt()
        self.omega0 = torch.where((nb > 0) & (nc > 0), nc / nb, 1.0)

    def set_values(self, val):
        lp = self.lp
        self.A = torch.sparse_csr_tensor(self.a_ptr, lp.col, val, (lp.m, lp.n))
        self.At = torch.sparse_csr_tensor(self.t_ptr, self.t_col, val[self.t_order], (lp.n, lp.m))

    def m_sum(self, v):
        return v.sum()[None] if self.k == 1 else _segment_sum(v, self.mlen)

    def n_sum(self, v):
        return v.sum()[None] if self.k == 1 else _segment_sum(v, self.nlen)

    def on_m(self, s):
        return s if self.k == 1 else s[self.lp.lp_of_row]

    def on_n(self, s):
        return s if self.k == 1 else s[self.lp.lp_of_col]

    def _power(self):
        v = 1.0 / self.on_n(self.nlen.double().sqrt()).expand(self.lp.n)
        lam = before = torch.zeros(self.k, device=v.device, dtype=torch.float64)
        live = torch.ones(self.k, device=v.device, dtype=torch.bool)
        for it in range(200):
            w = self.At @ (self.A @ v)
            q, norm = self.n_sum(v * w), self.n_sum(w * w).sqrt()
            lam = torch.where(live, q, lam)
            if it:
                live = live & ~((q - before).abs() <= 1e-10 * q)
            before = q
            v = w / self.on_n(norm)
            if it % 16 == 15 and not bool(live.any()):
                break
        return lam.sqrt()

    def _norms(self, x, y, ax, aty, x0, y0):
        rp, rd = self.b - ax, torch.clamp(self.c - aty, max=0.0)
        return dict(s1=self.m_sum(rp * rp), s2=self.n_sum(rd * rd), p=self.n_sum(self.c * x),
                    d=self.m_sum(self.b * y), u1=self.m_sum((rp / self.d_r) ** 2),
                    u2=self.n_sum((rd / self.d_c) ** 2), dx=self.n_sum((x - x0) ** 2).sqrt(),
                    dy=self.m_sum((y - y0) ** 2).sqrt())

    def iterate(self, eps, max_iter, rule="averaged"):
        """Until every LP meets the test at eps, or max_iter: the state, and
        per LP the iterations and the returned (scaled) x and y."""
        lp, F = self.lp, 64
        one = torch.ones(self.k, device=lp.b.device, dtype=torch.float64)
        x, y, ax = torch.zeros_like(self.c), torch.zeros_like(self.b), torch.zeros_like(self.b)
        xa, ya, axa, x0, y0, ax0 = x, y, ax, x, y, ax
        out_x, out_y = x, y
        omega, eta = self.omega0, self.eta
        nb, nc = self.m_sum(lp.b ** 2).sqrt(), self.n_sum(lp.c ** 2).sqrt()
        kkt_last = (omega ** 2 * self.m_sum(self.b ** 2) +
                    self.n_sum(torch.clamp(self.c, max=0.0) ** 2) / omega ** 2).sqrt()
        kkt_prev, t, eta_sum = kkt_last, 0 * one, 0 * one
        pid_sum, pid_prev = 0 * one, 0 * one
        live, iters = one > 0, torch.zeros(self.k, device=one.device, dtype=torch.int64)
        k = 0
        while k < max_iter:
            tau_n, sig_m = self.on_n(eta / omega), self.on_m(eta * omega)
            xn = torch.clamp(x - tau_n * (self.c - self.At @ y), min=0.0)
            h = self.A @ xn
            yn = y + sig_m * (self.b - 2 * h + ax)
            k += 1
            if rule.startswith("halpern"):
                lam = (t + 1) / (t + 2)
                ln, lm = self.on_n(lam), self.on_m(lam)
                xa, ya, axa = xn, yn, h
                x = ln * (2 * xn - x) + (1 - ln) * x0
                y = lm * (2 * yn - y) + (1 - lm) * y0
                ax = lm * (2 * h - ax) + (1 - lm) * ax0
            elif rule == "adaptive":
                dx, dy = xn - x, yn - y
                cross = self.m_sum(dy * (self.A @ dx)).abs()
                top = omega * self.n_sum(dx * dx) + self.m_sum(dy * dy) / omega
                most = torch.where(cross > 0, top / (2 * cross), math.inf)
                nxt = torch.minimum((1 - (k + 1.0) ** -0.3) * most, (1 + (k + 1.0) ** -0.6) * eta)
                if bool(eta <= most):
                    eta_sum = eta_sum + eta
                    w = eta / eta_sum
                    xa, ya, axa = xa + (xn - xa) * w, ya + (yn - ya) * w, axa + (h - axa) * w
                    x, y, ax = xn, yn, h
                eta = nxt
            else:
                w = 1 / (t + 1)
                wn, wm = self.on_n(w), self.on_m(w)
                xa, ya, axa = xa + (xn - xa) * wn, ya + (yn - ya) * wm, axa + (h - axa) * wm
                x, y, ax = xn, yn, h
            t = t + 1
            if k % F and k < max_iter:
                continue
            both = [self._norms(x, y, ax, self.At @ y, x0, y0), self._norms(xa, ya, axa, self.At @ ya, x0, y0)]
            met = [(q["u1"].sqrt() <= eps * (1 + nb)) & (q["u2"].sqrt() <= eps * (1 + nc)) &
                   ((q["p"] - q["d"]).abs() <= eps * (1 + q["p"].abs() + q["d"].abs())) for q in both]
            iters = torch.where(live, k, iters)
            ends = live & (met[0] | met[1] | (torch.full_like(live, k >= max_iter)))
            avg = met[1] & ~met[0]
            out_x = torch.where(self.on_n(ends), torch.where(self.on_n(avg), xa, x), out_x)
            out_y = torch.where(self.on_m(ends), torch.where(self.on_m(avg), ya, y), out_y)
            live = live & ~ends
            if not bool(live.any()):
                break
            kkt = [(omega ** 2 * q["s1"] + q["s2"] / omega ** 2 + (q["p"] - q["d"]) ** 2).sqrt() for q in both]
            cand = kkt[1] < kkt[0]
            pick = lambda f: torch.where(cand, both[1][f], both[0][f])  # noqa: E731
            kc, dx, dy = torch.minimum(*kkt), pick("dx"), pick("dy")
            again = (kc <= 0.2 * kkt_last) | ((kc <= 0.8 * kkt_last) & (kc > kkt_prev)) | (t >= 0.36 * k)
            kkt_prev = kc
            moved = again & (dx > 1e-10) & (dy > 1e-10)
            if rule.endswith("pid"):
                e = (dy / dx).log() - omega.log()
                pid_sum = torch.where(moved, pid_sum + e, pid_sum)
                new = (omega.log() + 0.99 * e + 0.01 * pid_sum).exp()
                pid_prev = torch.where(moved, e, pid_prev)
            else:
                new = (0.5 * (dy / dx).log() + 0.5 * omega.log()).exp()
            omega = torch.where(moved, new, omega)
            kkt_last = torch.where(again, kc, kkt_last)
            t, eta_sum = torch.where(again, 0 * t, t), torch.where(again, 0 * eta_sum, eta_sum)
            an, am = self.on_n(again), self.on_m(again)
            cn, cm = an & self.on_n(cand), am & self.on_m(cand)
            x, y, ax = torch.where(cn, xa, x), torch.where(cm, ya, y), torch.where(cm, axa, ax)
            x0, y0, ax0 = torch.where(an, x, x0), torch.where(am, y, y0), torch.where(am, ax, ax0)
        return dict(x=x, y=y, x_avg=xa, y_avg=ya, x_last=x0, y_last=y0, Ax=ax, iters=iters,
                    out_x=out_x, out_y=out_y)

    def z(self, y):
        return torch.clamp(self.c - self.At @ y, min=0.0)

    def solution(self, x, y):
        return dict(x=self.d_c * x, y=self.d_r * y, z=self.z(y) / self.d_c)

    def least_squares(self, rhs, w, on, tol):
        """Conjugate gradients on the normal equations of the columns `on`, per LP."""
        r = rhs - on * (self.At @ (self.A @ w))
        p, rr, stop = r, self.n_sum(r * r), tol ** 2 * self.n_sum(rhs * rhs)
        live = rr > stop
        for it in range(5000):
            q = on * (self.At @ (self.A @ p))
            pq = self.n_sum(p * q)
            live = live & (pq > 0)
            a = self.on_n(torch.where(live, rr / pq, 0.0))
            w, r = w + a * p, r - a * q
            new = self.n_sum(r * r)
            p = torch.where(self.on_n(live), r + self.on_n(new / rr) * p, p)
            live, rr = live & (new > stop), torch.where(live, new, rr)
            if it % 16 == 15 and not bool(live.any()):
                break
        return w


def _centered(x, z):
    mu = torch.clamp((x * z).sum() / x.numel(), min=1e-6)
    xp, zp, d = torch.clamp(x, min=1e-6), torch.clamp(z, min=1e-6), 1e-4
    move = lambda target, v: torch.minimum(torch.maximum(target, v - d), v + d)  # noqa: E731
    x_first = move(mu / zp, xp)
    z_first = move(mu / xp, zp)
    less = xp < zp
    return (torch.where(less, x_first, move(mu / z_first, xp)),
            torch.where(less, move(mu / x_first, zp), z_first), mu)


def exact(case, seed):
    kind = case["kind"]
    if kind == "center":
        st = prepare(case, seed)
        xw, zw, mu = _centered(st["x"], st["z"])
        return [xw, zw, mu[None]]
    lp, gen = _inputs(case, seed)
    p = _Plain(lp)
    if kind == "create":
        return dict(D_r=p.d_r, D_c=p.d_c, sigma_max=float(p.sigma), omega0=float(p.omega0))
    if kind == "batch":
        r = p.iterate(*((0.0, case["iters"]) if case["iters"] else (EPS, MAX_ITER)))
        out = p.solution(r["out_x"], r["out_y"])
        if case["precision"] == "fp32":
            out.pop("z")
        return dict(out, iters=None)
    if kind == "autograd":
        g = torch.randn(lp.n, generator=gen, device="cuda", dtype=torch.float64)
        r = p.iterate(EPS, MAX_ITER)
        on = (r["out_x"] > p.z(r["out_y"])).double()
        w = p.least_squares(on * (p.At @ p.b), on * r["out_x"], on, 1e-12)
        x = p.d_c * w
        p.set_values(lp.val)
        w = p.least_squares(on * g, torch.zeros_like(g), on, 1e-12)
        return dict(x=x, grad_b=p.A @ w)
    if kind == "iterate":
        r = p.iterate(0.0, case["iters"], case["rule"])
        return {k: r[k] for k in ("x", "y", "x_avg", "y_avg", "x_last", "y_last", "Ax")}
    r = p.iterate(*((0.0, 64) if kind == "finish" else (EPS, MAX_ITER)))
    out = p.solution(r["out_x"], r["out_y"])
    if kind == "solve":
        return dict(out, iters=None)
    xw, zw, mu = _centered(r["out_x"], p.z(r["out_y"]))
    return dict(out, x_ws=xw, y_ws=r["out_y"], z_ws=zw, mu=float(mu))
