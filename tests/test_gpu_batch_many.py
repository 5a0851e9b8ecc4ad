"""A batch of more small LPs than a grid has blocks in y (65,535 for two matrices
each): every copy of an LP gets the bits of the first one."""
import numpy as np
import pytest

from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("copies", [8191, 8192, 8250])  # 32,764, 32,768 and 33,000 LPs
def test_tens_of_thousands_of_lps(copies, precision):
    B.build()
    lps = [lpgen.planted_lp(3, 7, nnz_per_col=2, seed=s) for s in range(4)]

    def tiled(k):
        f = {"m": np.int32, "n": np.int32, "row_ptr": np.int32, "col": np.int32, "val": float, "b": float, "c": float}
        return {q: np.tile(np.concatenate([np.atleast_1d(getattr(lp, q)) for lp in lps]).astype(t), k) for q, t in f.items()}

    out = []
    for k in (1, copies):
        with pdhg.BatchSolver(arrays=tiled(k), precision=precision) as s:
            s.solve(0.0, 100)
            got = s.get()
            pol = s.polish()
            adj = s.adjoint(np.ones(s.n))
            out.append((got["x"], got["y"], pol["x"], adj["grad_b"]))
    for a, b in zip(*out):
        np.testing.assert_array_equal(b.reshape(copies, -1), np.broadcast_to(a, (copies, a.size)))
