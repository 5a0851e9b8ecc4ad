"""Large matrices in slices (a warp per slice of up to 32 rows sorted in windows
of 64) against the tile kernels, which a forced tile capacity asks for: rows at
the edges of the classes (24, 48 or 96 nonzeros with 1, 2 or 4 lanes per short
row, 128 with 8 lanes, a warp above), empty rows, last windows of 1 row, tails of
0 to 3 steps; and matrices that keep the tiles.

Tolerances as in the other parity tests: float64 states 1e-9 relative in the
infinity norm (the sums run in another order, about 1e-15 per product, over 100
iterations of a nonexpansive map).  Float32 half-steps keep the tiles.  The adaptive step
feeds its sums back into the step length, which is no such map (two capacities of
the tile kernels drift apart as fast): 10 attempts instead of 100."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu

SLICED = 64


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def rel_inf(a, b):
    a, b = np.asarray(a, float), np.asarray(b, float)
    return float(np.max(np.abs(a - b)) / max(1e-300, np.max(np.abs(b))))


def rows_lp(lengths, n, seed):
    """One row per entry of `lengths` at random columns, planted optimum."""
    rng = np.random.default_rng(seed)
    lengths = np.asarray(lengths)
    m, nnz = lengths.size, int(lengths.sum())
    ptr = np.concatenate([[0], np.cumsum(lengths)])
    # distinct columns of a row: a random start and a stride coprime to n (n prime)
    k = np.arange(nnz) - np.repeat(ptr[:-1], lengths)
    start, stride = rng.integers(0, n, m), rng.integers(1, n, m)
    cols = (np.repeat(start, lengths) + k * np.repeat(stride, lengths)) % n
    A = sp.csr_matrix((rng.standard_normal(nnz), cols, ptr), shape=(m, n))
    A.sort_indices()
    x = rng.uniform(0.5, 2, n) * (rng.random(n) < 0.3)
    z = np.where(x > 0, 0.0, rng.uniform(0.5, 2, n))
    b, c = A @ x, A.T @ rng.standard_normal(m) + z
    return lpgen.LP(m, n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, b, c)


def lengths(m, seed):
    """Runs of 32 equal lengths from the edges of every class, long ones rare."""
    rng = np.random.default_rng(seed)
    pool = [0, 1, 2, 3, 4, 5, 7, 8, 23, 24, 25, 47, 48, 49, 95, 96, 97, 127, 128, 129, 255, 256, 257, 600]
    p = np.array([1.0] * 16 + [0.5] + [0.2] * 6 + [0.05])
    return np.repeat(rng.choice(pool, size=m // 32 + 1, p=p / p.sum()), 32)[:m]


MAKERS = {  # 4, 2 and 1 lanes per short row of A; A^T's rows follow
    "lanes_4": lambda: rows_lp(lengths(14017, 1), 10007, 1),
    "lanes_2": lambda: rows_lp(lengths(20033, 2), 30011, 2),
    "lanes_1": lambda: rows_lp(lengths(44993, 3), 60013, 3),
    "planted": lambda: lpgen.planted_lp(33_001, 82_507, seed=5),
    "transport": lambda: lpgen.transportation_lp(417, 431),  # 14 steps a row
}


@pytest.mark.parametrize("method", ["averaged", "halpern", "adaptive"])
@pytest.mark.parametrize("name", list(MAKERS))
def test_states_match_the_tile_kernels(name, method):
    lp = MAKERS[name]()
    kw, iters = {}, 10 if method == "adaptive" else 100
    kw.update({"step_rule": "adaptive"} if method == "adaptive" else {"method": method})
    with pdhg.Solver.from_lp(lp, **kw) as s, pdhg.Solver.from_lp(lp, tile_nnz=2044, **kw) as t:
        assert s.schedule()["a_variant"] == s.schedule()["at_variant"] == SLICED
        assert t.schedule()["a_variant"] != SLICED and t.schedule()["at_variant"] != SLICED
        sa, sb = s.scaling()["sigma_max"], t.scaling()["sigma_max"]
        assert abs(sa - sb) < 1e-12 * sb
        for q in (s, t):
            assert q.solve(0.0, iters) == pdhg.PDHG_MAX_ITER
        a, b = s.state(), t.state()
        for k in ("x", "y", "x_avg", "y_avg"):
            assert rel_inf(a[k], b[k]) < 1e-9, k


@pytest.mark.parametrize("name,rows", [
    ("too_long", np.r_[3000, np.full(21000, 17)]),  # 94 steps, 0.36 million nonzeros
    ("too_ragged", np.where(np.arange(96000) % 64 == 0, 24, 1)),  # padded above 2 x
])
def test_matrices_that_keep_the_tiles(name, rows):
    lp = rows_lp(rows, 30011, 4)
    with pdhg.Solver.from_lp(lp) as s:
        assert s.schedule()["a_variant"] != SLICED and s.schedule()["at_variant"] == SLICED


def test_float32_half_steps_keep_the_order_of_the_tiles():
    lp = MAKERS["planted"]()
    out = []
    for kw in ({"autotune": 0}, {"tile_nnz": 2044}):  # the same schedules
        with pdhg.Solver.from_lp(lp, precision="fp32", **kw) as s:
            assert s.schedule()["a_variant"] != SLICED and s.schedule()["at_variant"] != SLICED
            assert s.solve(0.0, 64) == pdhg.PDHG_MAX_ITER
            out.append(s.state())
    for k in ("x", "y", "x_avg", "y_avg"):
        np.testing.assert_array_equal(out[0][k], out[1][k], err_msg=k)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("method", ["averaged", "halpern", "adaptive"])
@pytest.mark.parametrize("name", ["lanes_4", "lanes_1", "planted"])
def test_a_non_finite_entry_reaches_its_own_rows_only(name, method, bad):
    """Entry 0 of y (then of x) infinite or NaN: the products, the next iterate
    and the returned solution are non-finite where the tile kernels' are, and
    the rest agrees to 1e-9 as above."""
    lp = MAKERS[name]()
    kw = {"step_rule": "adaptive"} if method == "adaptive" else {"method": method}
    with pdhg.Solver.from_lp(lp, **kw) as s, pdhg.Solver.from_lp(lp, tile_nnz=2044, **kw) as t:
        assert s.schedule()["a_variant"] == s.schedule()["at_variant"] == SLICED
        s.solve(0.0, 8)
        good = s.state()
        for field in ("y", "x"):
            out = []
            for q in (s, t):
                st = {k: np.array(v) if isinstance(v, np.ndarray) else v for k, v in good.items()}
                st[field][0] = bad
                st = {k: v for k, v in st.items() if not k.startswith("Ax")}  # products from the state
                q.set_state(st)
                before = {k: v for k, v in q.state().items() if k.startswith("Ax")}
                g = q.get()
                q.solve(0.0, 9)
                out.append({**before, **{"get_" + k: g[k] for k in "xyz"}, **{k: q.state()[k] for k in ("x", "y")}})
            for k in out[0]:
                a, b = out[0][k], out[1][k]
                fin = np.isfinite(b)
                np.testing.assert_array_equal(np.isfinite(a), fin, err_msg=f"{field} {k}")
                assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[~fin] > 0, b[~fin] > 0), k
                assert fin.mean() > 0.5 and rel_inf(a[fin], b[fin]) < 1e-9, (field, k)
