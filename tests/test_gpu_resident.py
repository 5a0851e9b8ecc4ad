"""LPs solved on chip (a thread-block cluster per LP) against the oracle and
against the tile kernels, at the edges of the layout: rows of 0, 1, 24, 25,
256, 257 and 4096 nonzeros (the three row classes and their limit), last
slices of 1 and 32 rows, more rows than columns, clusters of 1 to 16.

Tolerances as in the other parity tests: float64 states 1e-9 relative in the
infinity norm (the sums run in another order, about 1e-15 per product, over
200 iterations of a nonexpansive map); float32-mixed states 1e-4."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import pdhg_oracle as O
from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu

KEYS = ["x", "y", "x_avg", "y_avg", "x_last", "y_last", "Ax", "Ax_avg", "Ax_last"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def rel_inf(a, b):
    a, b = np.asarray(a, float), np.asarray(b, float)
    return float(np.max(np.abs(a - b)) / max(1e-300, np.max(np.abs(b))))


def rows_lp(lengths, n, seed):
    """One row per entry of `lengths`, planted optimum."""
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lengths]
    ptr = np.concatenate([[0], np.cumsum([c.size for c in cols])])
    val = rng.standard_normal(int(ptr[-1]))
    A = sp.csr_matrix((val, np.concatenate(cols).astype(int) if cols else [], ptr), shape=(len(lengths), n))
    x = rng.uniform(0.5, 2, n) * (rng.random(n) < 0.3)
    z = np.where(x > 0, 0.0, rng.uniform(0.5, 2, n))
    b, c = A @ x, A.T @ rng.standard_normal(len(lengths)) + z
    return lpgen.LP(len(lengths), n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, b, c)


MAKERS = {
    "tiny": lambda: lpgen.planted_lp(3, 7, nnz_per_col=2, seed=0),
    "short_edge": lambda: rows_lp([24] * 33 + [25] * 5 + [0, 1, 0], 64, 1),
    "mid_edge": lambda: rows_lp([256] * 3 + [257] * 2 + [3] * 40, 300, 2),
    "longest": lambda: rows_lp([4096, 4095, 31] + [4] * 61, 5000, 3),
    "tall": lambda: rows_lp(list(range(1, 90)) + [2] * 700, 97, 4),
    "planted": lambda: lpgen.planted_lp(331, 829, seed=5),
    "wide_cluster": lambda: lpgen.planted_lp(2311, 5777, seed=6),
    "transport": lambda: lpgen.transportation_lp(31, 44),
}


def run(lp, iters, **kw):
    """A float32-mixed LP runs in a batch of its own: alone it keeps the tile
    kernels (their order of addition)."""
    if kw.get("precision") == "fp32":
        kw = dict(kw, method=0, omega_rule=0)  # (batches run the averaged iteration)
        with pdhg.BatchSolver([lp], **kw) as s:
            before = s.launch_count()
            s.solve(0.0, iters)
            launches = s.launch_count() - before
            return s.get(), [], launches
    with pdhg.Solver.from_lp(lp, **kw) as s:
        before = s.launch_count()
        assert s.solve(0.0, iters) == pdhg.PDHG_MAX_ITER
        return s.state(), s.log(), s.launch_count() - before


@pytest.mark.parametrize("name", list(MAKERS))
def test_float64_iterates_match_oracle(name):
    lp = MAKERS[name]()
    st, lg, launches = run(lp, 100)
    assert launches < 10  # one launch, not one per half-step
    r = O.solve(lp, 0.0, 100)
    for k in KEYS[:6]:
        assert rel_inf(st[k], getattr(r.state, k)) < 1e-9, k
    assert [(e["k"], e["restart"], e["cand"]) for e in lg] == \
           [(e["k"], e["restart"], e["cand"]) for e in r.log]


@pytest.mark.parametrize("method,rule,precision,tol", [
    ("averaged", "smooth", "fp64", 1e-9), ("halpern", "pid", "fp64", 1e-9), ("averaged", "smooth", "fp32", 1e-4)])
@pytest.mark.parametrize("name", list(MAKERS))
def test_states_match_the_tile_kernels(name, precision, tol, method, rule):
    """200 iterations: an odd last chunk, three evaluations, restarts; the tile
    kernels are asked for by a forced tile capacity."""
    lp = MAKERS[name]()
    kw = dict(precision=precision, method=method, omega_rule=rule)
    a, la, n_a = run(lp, 200, **kw)
    b, lb, n_b = run(lp, 200, tile_nnz=2044, **kw)
    assert n_a < 10 < n_b
    # the two candidates of an LP that float32 has already solved to its last
    # digit ("tall" at 192) differ by rounding alone: decisions are float64's
    if precision == "fp64":
        assert [(e["k"], e["restart"], e["cand"]) for e in la] == \
               [(e["k"], e["restart"], e["cand"]) for e in lb]
    for k in KEYS if precision == "fp64" else KEYS[:2]:
        assert rel_inf(a[k], b[k]) < tol, k


def test_a_single_float32_lp_keeps_the_order_of_the_tile_kernels():
    lp = MAKERS["planted"]()
    a, _, n = run(lp, 64, precision="fp64")
    assert n < 10
    out = []
    for kw in ({"autotune": 0}, {"tile_nnz": 2044}):  # the same schedule
        with pdhg.Solver.from_lp(lp, precision="fp32", **kw) as s:
            before = s.launch_count()
            assert s.solve(0.0, 64) == pdhg.PDHG_MAX_ITER
            assert s.launch_count() - before > 64
            out.append(s.state())
    for k in KEYS:
        np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=k)


def test_rows_past_the_limit_take_the_tile_kernels():
    lp = rows_lp([4097] + [3] * 50, 5000, 7)
    st, _, launches = run(lp, 64)
    assert launches > 64
    assert rel_inf(st["x"], O.solve(lp, 0.0, 64).state.x) < 1e-9


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-4)])
def test_batch_of_every_cluster_size(precision, tol):
    """LPs from 3 x 7 to 2300 x 5750 in one batch: each LP its own cluster size,
    several launches side by side; resumed from a stop between evaluations."""
    lps = [lpgen.planted_lp(3, 7, nnz_per_col=2, seed=0), MAKERS["tall"](), MAKERS["mid_edge"](), lpgen.planted_lp(2300, 5750, seed=1)]
    lps += [lpgen.planted_lp(m, int(2.5 * m), seed=m) for m in (40, 150, 400, 900)]
    out = []
    for persistent in (0, 1):  # the persistent form runs on the tile kernels
        with pdhg.BatchSolver(lps, precision=precision, persistent=persistent) as s:
            s.solve(0.0, 100)
            s.solve(0.0, 200)
            out.append(s.get())
    a, b = out
    assert np.array_equal(a["iters"], b["iters"])
    assert rel_inf(a["x"], b["x"]) < tol and rel_inf(a["y"], b["y"]) < tol


def test_a_stop_between_evaluations_changes_nothing():
    lp = MAKERS["planted"]()
    with pdhg.Solver.from_lp(lp) as s:
        s.solve(0.0, 192)
        ref = s.state()
    with pdhg.Solver.from_lp(lp) as s:
        for k in (1, 37, 100, 192):
            s.solve(0.0, k)
        got = s.state()
    for k in KEYS:
        np.testing.assert_array_equal(got[k], ref[k], err_msg=k)


def test_polish_and_adjoint_match_the_tile_kernels():
    """Conjugate gradients on chip, cut down to the active columns, against the
    tile kernels': LPs of every row class, more rows than columns, no active
    column at all (b = 0), and one large enough for a wide cluster.  Both stop
    at a relative residual of 1e-12 of normal equations of condition up to 1e4
    or so: 1e-8 relative."""
    lps = [MAKERS[k]() for k in ("planted", "short_edge", "mid_edge", "tall", "wide_cluster")]
    lps.append(lpgen.planted_lp(30, 80, seed=3, n_pos=0))
    g = np.random.default_rng(0).standard_normal(sum(lp.n for lp in lps))
    out = []
    for kw in ({}, {"tile_nnz": 2044}):
        with pdhg.BatchSolver(lps, **kw) as s:
            s.solve(1e-4, 20_000)
            before = s.launch_count()
            p = s.polish()
            out.append((p["active"], p["x"], s.adjoint(g)["grad_b"], s.launch_count() - before, p["cg_iters"]))
            if not kw:  # a second active set in the same context
                s.set_rhs(np.concatenate([lp.b for lp in lps]), np.concatenate([lp.c for lp in lps]))
                s.solve(1e-4, 20_000)
                np.testing.assert_array_equal(s.polish()["x"], p["x"])
                np.testing.assert_array_equal(s.adjoint(g)["grad_b"], out[0][2])
    a, b = out
    np.testing.assert_array_equal(a[0], b[0])
    assert a[0][-1] == 0 and a[4][-1] == 0
    assert a[3] < b[3]
    assert rel_inf(a[1], b[1]) < 1e-8
    # the adjoint is A_B (A_B^T A_B)^-1 g: with more active columns than rows
    # ("mid_edge") that matrix is singular and no solution exists to compare
    first = np.concatenate([[0], np.cumsum([lp.m for lp in lps])])
    defined = [i for i, lp in enumerate(lps) if a[0][i] <= lp.m]
    assert len(defined) == len(lps) - 1
    for i in defined:
        u, v = a[2][first[i]:first[i + 1]], b[2][first[i]:first[i + 1]]
        assert np.array_equal(u, v) or rel_inf(u, v) < 1e-8, i
