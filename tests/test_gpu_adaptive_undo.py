"""Rejected attempts of the adaptive step within a run of attempts: the attempt
after a rejected one reads the saved state in place of the new one, on tiles (also
with rows split across tiles) and on slices.

Tolerance as in the other adaptive tests against the oracle: 1e-9 relative in the
infinity norm."""
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


def _setup_from(s, lp):
    sc = s.scaling()
    Dr, Dc = np.array(sc["D_r"], dtype=np.float64), np.array(sc["D_c"], dtype=np.float64)
    A = O.as_csr(lp.m, lp.n, lp.row_ptr, lp.col, lp.val)
    At = (sp.diags(Dr) @ A @ sp.diags(Dc)).tocsr()
    b, c = np.asarray(lp.b, float), np.asarray(lp.c, float)
    return O.Setup(A, b, c, Dr, Dc, At, Dr * b, Dc * c, sc["sigma_max"], sc["power_iters"],
                   sc["eta"], sc["omega0"])


@pytest.mark.parametrize("maker,tile_nnz", [
    (lambda: lpgen.planted_lp(200, 500, seed=0), 0),
    (lambda: lpgen.planted_lp(200, 500, seed=0), 20),
    (lambda: lpgen.planted_lp(8000, 20000, seed=3), 0),
])
@pytest.mark.parametrize("attempts", [2, 3, 10])
def test_attempts_after_a_rejected_one(maker, tile_nnz, attempts):
    lp = maker()
    with pdhg.Solver.from_lp(lp, step_rule="adaptive", tile_nnz=tile_nnz) as s:
        S = _setup_from(s, lp)
        assert s.solve(1e-12, 64) == pdhg.PDHG_MAX_ITER  # away from the zero state
        o = O.solve(lp, 1e-12, 64, opts=O.Options(step_rule="adaptive"), S=S).state
        now, step = s.state(), s.step_state()
        s.set_state(dict(now, step_eta=100.0 * step["step_eta"], eta_sum=step["eta_sum"]))
        o.eta = 100.0 * step["step_eta"]
        r = O.solve(lp, 1e-12, 64 + attempts, opts=O.Options(step_rule="adaptive"), S=S, state=o)
        assert r.state.step_rejects >= 1
        assert s.solve(1e-12, 64 + attempts) == pdhg.PDHG_MAX_ITER
        st = s.state()
        assert s.step_state()["step_rejects"] == r.state.step_rejects
    for k in ("x", "y", "x_avg", "y_avg"):
        a, b = st[k], getattr(r.state, k)
        assert np.max(np.abs(a - b)) < 1e-9 * max(1e-300, np.max(np.abs(b))), k
