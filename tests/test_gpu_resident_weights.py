"""On-chip solves with more than 64 iterations between evaluations: the averaging
and Halpern weights are taken 64 at a time.  Against the oracle after 430
iterations, clusters of 1, 4 and 16 CTAs; float64 states 1e-9 relative as in the
other parity tests."""
import numpy as np
import pytest

from oracle import pdhg_oracle as O
from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["averaged", "halpern"])
@pytest.mark.parametrize("freq", [63, 64, 65, 128, 200])
@pytest.mark.parametrize("m", [30, 200, 1500])
def test_weights_between_evaluations(m, freq, method):
    B.build()
    lp = lpgen.planted_lp(m, 5 * m // 2, seed=m)
    r = O.solve(lp, 0.0, 430, opts=O.Options(method=method, eval_freq=freq))
    with pdhg.Solver.from_lp(lp, method=method, eval_freq=freq) as s:
        before = s.launch_count()
        assert s.solve(0.0, 430) == pdhg.PDHG_MAX_ITER
        assert s.launch_count() - before < 10
        st = s.state()
    for k in ("x", "y", "x_avg", "y_avg"):
        a, b = st[k], getattr(r.state, k)
        assert np.max(np.abs(a - b)) < 1e-9 * np.max(np.abs(b)), k
