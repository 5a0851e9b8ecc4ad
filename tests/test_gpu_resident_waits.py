"""On-chip solves whose clusters have warps, or whole CTAs, without rows of a
matrix: such warps are not held back by the vectors they would wait for.  The
same iterations run in one call and in many must give the same bits, and no
wait may run out."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def few_rows_lp(m, n, per_row, seed, transposed=False):
    """m rows of per_row nonzeros each over n columns (or the transpose)."""
    rng = np.random.default_rng(seed)
    cols = np.concatenate([np.sort(rng.choice(n, size=per_row, replace=False)) for _ in range(m)])
    A = sp.csr_matrix((rng.standard_normal(m * per_row), cols, np.arange(m + 1) * per_row), shape=(m, n))
    if transposed:
        A = sp.csr_matrix(A.T)
    x = rng.uniform(0.5, 2, A.shape[1]) * (rng.random(A.shape[1]) < 0.3)
    z = np.where(x > 0, 0.0, rng.uniform(0.5, 2, A.shape[1]))
    b, c = A @ x, A.T @ rng.standard_normal(A.shape[0]) + z
    A.sort_indices()
    return lpgen.LP(A.shape[0], A.shape[1], A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, b, c)


MAKERS = {
    "idle_warps": lambda: lpgen.planted_lp(200, 500, seed=0),            # 12 of 16 warps of a CTA
    "ctas_without_rows": lambda: few_rows_lp(6, 5000, 4000, 1),          # 6 slices of A~ on 16 CTAs
    "ctas_without_columns": lambda: few_rows_lp(6, 5000, 4000, 2, True),  # 6 slices of A~^T
}


@pytest.mark.parametrize("method", ["averaged", "halpern"])
@pytest.mark.parametrize("name", list(MAKERS))
def test_long_runs_in_one_call_and_in_many(name, method):
    lp = MAKERS[name]()
    out = []
    for step in (20_000, 500):
        with pdhg.Solver.from_lp(lp, method=method) as s:
            before = s.launch_count()
            for k in range(step, 20_001, step):
                assert s.solve(0.0, k) == pdhg.PDHG_MAX_ITER
            assert s.launch_count() - before <= 20_000 // step + 20
            out.append((s.scaling()["sigma_max"], s.state()))
    assert out[0][0] == out[1][0]
    for k in ("x", "y", "x_avg", "y_avg"):
        np.testing.assert_array_equal(out[0][1][k], out[1][1][k], err_msg=k)


@pytest.mark.parametrize("name", list(MAKERS))
def test_power_iteration_many_times(name):
    lp = MAKERS[name]()
    sigma = set()
    for _ in range(10):
        with pdhg.Solver.from_lp(lp, power_rel_tol=0.0, power_max_iter=2000) as s:
            sigma.add(s.scaling()["sigma_max"])
    assert len(sigma) == 1


def gives_up(create, call=None):
    """create() or call(solver) ends with PDHG_TIMEOUT; the GPU stays usable."""
    if call is None:
        with pytest.raises(pdhg.PDHGError) as e:
            create()
        assert e.value.status == pdhg.PDHG_TIMEOUT
    else:
        with create() as s:
            for _ in range(2):
                call(s)
    lp = lpgen.planted_lp(200, 500, seed=1)
    with pdhg.Solver.from_lp(lp) as s:
        assert s.solve(1e-4, 20_000) == pdhg.PDHG_CONVERGED


# clusters of 2, 4, 8 and 16 CTAs, and of CTAs without rows of a matrix
CLUSTERS = {f"planted_{m}": (lambda m=m: lpgen.planted_lp(m, 5 * m // 2, seed=m)) for m in (100, 200, 400, 900)}
CLUSTERS.update({k: v for k, v in MAKERS.items() if k != "idle_warps"})


@pytest.mark.parametrize("method", ["averaged", "halpern"])
@pytest.mark.parametrize("name", list(CLUSTERS))
def test_solve_whose_wait_runs_out(name, method):
    """options.wait_test makes each exchange expect 8 bytes that nobody sends
    (without a power iteration, which would give up first)."""
    lp = CLUSTERS[name]()

    def call(s):
        assert s.solve(1e-4, 1000) == pdhg.PDHG_TIMEOUT

    gives_up(lambda: pdhg.Solver.from_lp(lp, method=method, power_max_iter=0, wait_test=True, wait_limit_ms=5), call)


def test_batch_whose_waits_run_out():
    """LPs of every cluster size, one of a single CTA (which has no exchanges)."""
    lps = [lpgen.planted_lp(m, 5 * m // 2, seed=m) for m in (12, 200, 400, 800, 1600)]

    def call(s):
        assert s.solve(1e-4, 1000) == pdhg.PDHG_TIMEOUT
        assert list(s.lp_status) == [pdhg.PDHG_TIMEOUT] * len(lps)

    for precision in ("fp64", "fp32"):
        gives_up(lambda: pdhg.BatchSolver(lps, precision=precision, power_max_iter=0, wait_test=1, wait_limit_ms=5), call)


@pytest.mark.parametrize("name", list(CLUSTERS))
def test_power_iteration_whose_wait_runs_out(name):
    lp = CLUSTERS[name]()
    gives_up(lambda: pdhg.Solver.from_lp(lp, wait_test=True, wait_limit_ms=5))


def one_cta_lp(m=20, n=400, per_col=2):
    """Solved by one CTA, which has no exchanges; with every column active its
    conjugate gradients have enough work for two.  All data positive and c = 0:
    every entry of x moves off zero and none has a z."""
    rng = np.random.default_rng(7)
    rows = np.concatenate([rng.choice(m, size=per_col, replace=False) for _ in range(n)])
    A = sp.csr_matrix((rng.uniform(0.5, 1.5, n * per_col), (rows, np.repeat(np.arange(n), per_col))), shape=(m, n))
    A.sort_indices()
    return lpgen.LP(m, n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, A @ np.ones(n), np.zeros(n))


def test_polish_whose_wait_runs_out():
    lp = one_cta_lp()

    def call(s):
        s.solve(0.0, 64)
        with pytest.raises(pdhg.PDHGError) as e:
            s.polish()
        assert e.value.status == pdhg.PDHG_TIMEOUT

    gives_up(lambda: pdhg.BatchSolver([lp], wait_test=1, wait_limit_ms=5), call)
    with pdhg.BatchSolver([lp]) as s:
        s.solve(0.0, 64)
        assert s.polish()["active"][0] == lp.n
