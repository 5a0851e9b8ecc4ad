"""LPs whose layouts for the faster kernels (slices, on chip, on-chip conjugate
gradients) no longer fit in device memory take the tile kernels, which fit.  The
rest of the memory is held by one allocation meanwhile; how much each form needs
is read off a run with room to spare."""
import contextlib

import numpy as np
import pytest

from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import lpgen
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu

MB = 1 << 20


@contextlib.contextmanager
def only(free):
    """At most about `free` bytes of device memory left."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def held(make):
    """Device memory that make()'s solver holds (made once before, so that code is loaded)."""
    import torch
    make().close()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = make()
    n = before - torch.cuda.mem_get_info()[0]
    s.close()
    return n


def test_slices_without_room():
    B.build()
    lp = lpgen.planted_lp(300_000, 750_000, seed=1)
    tiles, sliced = (held(lambda: pdhg.Solver.from_lp(lp, **kw)) for kw in (dict(tile_nnz=2044), {}))
    assert sliced > tiles + 64 * MB
    with pdhg.Solver.from_lp(lp, tile_nnz=2044) as s:
        s.solve(0.0, 64)
        want = s.state()
    with only(sliced - 40 * MB):
        with pdhg.Solver.from_lp(lp) as s:
            sch = s.schedule()
            assert 64 not in (sch["a_variant"], sch["at_variant"]) or sch["a_variant"] != sch["at_variant"]
            s.solve(0.0, 64)
            got = s.state()
    for k in ("x", "y"):
        assert np.max(np.abs(got[k] - want[k])) < 1e-9 * np.max(np.abs(want[k]))
    with pdhg.Solver.from_lp(lp) as s:
        assert s.schedule()["a_variant"] == s.schedule()["at_variant"] == 64


def test_on_chip_layouts_without_room():
    B.build()
    lps = [lpgen.planted_lp(2000, 5000, seed=s) for s in range(8)]
    arrays = {q: np.tile(np.concatenate([np.atleast_1d(getattr(lp, q)) for lp in lps]), 30)
              for q in ("m", "n", "row_ptr", "col", "val", "b", "c")}  # 240 LPs, 6 million nonzeros

    def make(**kw):
        return pdhg.BatchSolver(arrays=arrays, **kw)

    def run(s):
        before = s.launch_count()
        s.solve(0.0, 64)
        n = s.launch_count() - before
        got = s.get()
        pol = s.polish(cg_tol=1e-9)
        s.adjoint(np.ones(s.n), cg_tol=1e-9)
        return got, pol["active"], n

    tiles, chip = held(lambda: make(tile_nnz=2044)), held(make)
    assert chip > tiles + 64 * MB
    with make() as s:
        want, active, n = run(s)
        assert n < 10
    with only(chip - 40 * MB):  # no room for the on-chip layout
        with make() as s:
            s.solve(0.0, 64)
            got = s.get()
    for k in ("x", "y"):
        assert np.max(np.abs(got[k] - want[k])) < 1e-9 * np.max(np.abs(want[k]))
    with make() as s:  # room for that, not for the conjugate gradients' (and the tile kernels' 8 vectors)
        s.solve(0.0, 64)
        with only(160 * MB):
            pol = s.polish(cg_tol=1e-9)
        np.testing.assert_array_equal(pol["active"], active)
        s.adjoint(np.ones(s.n), cg_tol=1e-9)
