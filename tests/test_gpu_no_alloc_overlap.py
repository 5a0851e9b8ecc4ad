"""Calls of pdhg_centered_point_noalloc share one static scratch, and calls that
overlap race for it: their results are undefined.  Calls that are serialised
after them must not be affected."""
import numpy as np
import pytest

from oracle import pdhg_oracle as O
from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu


def test_overlapping_calls_leave_later_ones_alone():
    import torch
    B.build()
    rng = np.random.default_rng(3)
    cases = []
    for n in (4097, 50_000, 300_001, 2_000_000):
        x = np.where(rng.random(n) < 0.3, rng.uniform(0, 2, n), 0.0)
        z = rng.uniform(0, 1e-3, n)
        t = [torch.as_tensor(v, device="cuda") for v in (x, z)]
        cases.append((x, z, t, [torch.empty_like(t[0]) for _ in range(2)], torch.empty(1, dtype=torch.float64, device="cuda")))
    streams = [torch.cuda.Stream() for _ in cases]
    torch.cuda.synchronize()
    for _ in range(200):
        for s, (_, _, t, o, mu) in zip(streams, cases):
            pdhg.centered_point_noalloc(*t, *o, mu, stream=s.cuda_stream)
    torch.cuda.synchronize()
    for x, z, t, o, mu in cases:
        for v in (*o, mu):
            v.fill_(float("nan"))
        pdhg.centered_point_noalloc(*t, *o, mu)
        torch.cuda.synchronize()
        ox, oz, omu = O.centered_start_point(x, z)
        # 2 million products added in another order, as in the tests of one call
        assert abs(mu.item() - omu) <= 1e-11 * omu
        for got, want in zip(o, (ox, oz)):
            assert np.max(np.abs(got.cpu().numpy() - want)) < 1e-9 * np.max(np.abs(want))
