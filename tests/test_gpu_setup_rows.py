"""The set-up's passes over the nonzeros (validation, transpose, scaled copies) on
matrices whose rows are hard to find from a nonzero's place: rows longer than a
warp's 256 nonzeros, long runs of empty rows, rows of one nonzero, a last warp
that is not full.  The spectral norm and ten iterations against the oracle's
(1e-9, as in the other parity tests); an invalid column or order anywhere in a
row is still found."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import pdhg_oracle as O
from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def rows_lp(lengths, n, seed=0):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(n, size=k, replace=False)) for k in lengths]
    ptr = np.concatenate([[0], np.cumsum(lengths)])
    A = sp.csr_matrix((rng.uniform(0.5, 2, int(ptr[-1])), np.concatenate(cols).astype(int), ptr),
                      shape=(len(lengths), n))
    b = A @ rng.uniform(0, 1, n)
    return lpgen.LP(len(lengths), n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, b,
                    rng.uniform(0, 1, n))


LENGTHS = {
    "one": [1],
    "ones": [1] * 700,
    "gaps": [3] + [0] * 5000 + [1] + [0] * 40 + [2] * 31 + [0] * 33 + [5],
    "long": [700] + [0] * 3 + [1] * 40 + [513, 255, 256, 257],
    "ends_empty": [0] * 100 + [7] * 73 + [0] * 100,
}


@pytest.mark.parametrize("name", list(LENGTHS))
def test_setup_matches_the_oracle(name):
    lp = rows_lp(LENGTHS[name], 800)
    S = O.setup(lp)
    with pdhg.Solver.from_lp(lp, tile_nnz=2044) as s:
        assert abs(s.scaling()["sigma_max"] - S.sigma_max) <= 1e-9 * S.sigma_max
        assert s.solve(0.0, 10) == pdhg.PDHG_MAX_ITER
        x, y = s.state()["x"], s.state()["y"]
    r = O.solve(lp, 0.0, 10, S=S)
    for a, b in ((x, r.state.x), (y, r.state.y)):
        assert np.max(np.abs(a - b)) <= 1e-9 * max(1e-300, np.max(np.abs(b)))


@pytest.mark.parametrize("at", [1, 255, 256, 257, 699])
def test_invalid_columns_are_found(at):
    lp = rows_lp(LENGTHS["long"], 800)
    for bad in (800, -1, int(lp.col[at - 1])):
        col = lp.col.copy()
        col[at] = bad
        with pytest.raises(pdhg.PDHGError):
            pdhg.Solver(lp.m, lp.n, lp.row_ptr, col, lp.val, lp.b, lp.c)
