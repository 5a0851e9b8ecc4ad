"""Small LPs solved on chip with 1, 2 and 4 lanes per short row (matrices of up to
90 rows per CTA whose rows average 6 and 12 nonzeros) against the tile kernels:
row counts around a slice of 8, 16 and 32 rows and around the limit, rows that do
not fill their lanes, empty rows, rows of the longer classes beside short ones.

Tolerances as in the other parity tests: float64 states 1e-9 relative in the
infinity norm (sums in another order over 100 iterations of a nonexpansive map),
float32-mixed solutions (of a batch of one LP: a float32 LP alone keeps the tile
kernels) 1e-4."""
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


def rows_lp(lengths, n, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lengths]
    ptr = np.concatenate([[0], np.cumsum([c.size for c in cols])])
    A = sp.csr_matrix((rng.standard_normal(int(ptr[-1])), np.concatenate(cols).astype(int), ptr),
                      shape=(len(lengths), n))
    x = rng.uniform(0.5, 2, n) * (rng.random(n) < 0.3)
    z = np.where(x > 0, 0.0, rng.uniform(0.5, 2, n))
    b, c = A @ x, A.T @ rng.standard_normal(len(lengths)) + z
    return lpgen.LP(len(lengths), n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, b, c)


def rel_inf(a, b):
    a, b = np.asarray(a, float), np.asarray(b, float)
    return float(np.max(np.abs(a - b)) / max(1e-300, np.max(np.abs(b))))


POOLS = {1: [0, 1, 3, 5, 9], 2: [0, 5, 7, 8, 13, 24], 4: [11, 12, 13, 23, 24, 25, 40]}


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-4)])
@pytest.mark.parametrize("lanes", [1, 2, 4])
@pytest.mark.parametrize("rows", [1, 7, 8, 9, 16, 17, 33, 90, 91, 181])
def test_states_match_the_tile_kernels(rows, lanes, precision, tol):
    pool = POOLS[lanes]
    lp = rows_lp(np.resize(pool[::-1], rows), 127, rows)
    out = []
    for tile_nnz in (0, 2044):
        if precision == "fp32":
            with pdhg.BatchSolver([lp], precision=precision, tile_nnz=tile_nnz) as s:
                s.solve(0.0, 100)
                out.append((s.get(), 0.0))
            continue
        with pdhg.Solver.from_lp(lp, precision=precision, tile_nnz=tile_nnz) as s:
            assert s.solve(0.0, 100) == pdhg.PDHG_MAX_ITER
            out.append((s.state(), s.scaling()["sigma_max"]))
    (a, sa), (b, sb) = out
    assert abs(sa - sb) <= 1e-12 * sb
    for k in ("x", "y", "x_avg", "y_avg") if precision == "fp64" else ("x", "y"):
        assert rel_inf(a[k], b[k]) < tol, k
