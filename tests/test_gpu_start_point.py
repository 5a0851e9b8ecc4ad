"""The no-allocation start point at the edges of its two forms (a cluster of
blocks up to 4096 entries, partial sums by many blocks above) and on special values, against
the oracle.  Tolerance: the sums of up to 70,000 positive products agree to
1e-12, so mu and the moved entries to 1e-11 relative."""
import numpy as np
import pytest

from oracle import pdhg_oracle as O
from paper_2603_03150_gb300 import build as B
from paper_2603_03150_gb300 import pdhg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()


def start_point(x, z, **kw):
    import torch
    xd, zd = torch.from_numpy(x).cuda(), torch.from_numpy(z).cuda()
    xo, zo, mu = torch.empty_like(xd), torch.empty_like(zd), torch.empty(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    pdhg.centered_point_noalloc(xd, zd, xo, zo, mu, **kw)
    torch.cuda.synchronize()
    return xo.cpu().numpy(), zo.cpu().numpy(), float(mu[0])


@pytest.mark.parametrize("n", [1, 31, 256, 257, 2047, 2048, 2049, 4096, 4097, 70001])
def test_sizes_around_the_forms(n):
    rng = np.random.default_rng(n)
    x = rng.uniform(0, 2, n) * (rng.random(n) < 0.5)
    z = np.where(x > 0, 1e-7 * rng.random(n), rng.uniform(0, 2, n))
    z[::7] = x[::7]  # ties: z moves first
    for _ in range(2):  # a second call finds the scratch as the first left it
        got = start_point(x, z)
        ox, oz, omu = O.centered_start_point(x, z)
        assert abs(got[2] - omu) <= 1e-12 * omu
        np.testing.assert_allclose(got[0], ox, rtol=1e-11)
        np.testing.assert_allclose(got[1], oz, rtol=1e-11)


def test_negative_zero_infinite_and_nan_entries():
    """Entry by entry as fmax / fmin define it: a NaN counts as alpha_min, an
    infinity stays; mu is given by mu_min (the sum is NaN)."""
    v = np.array([0.0, -0.0, 1e-300, 1e-7, 1e-6, 1.0, -1.0, 1e300, np.inf, -np.inf, np.nan])
    x, z = (a.ravel().copy() for a in np.meshgrid(v, v))
    got = start_point(x, z, mu_min=0.5)

    def move(t, w, d):
        return np.fmin(np.fmax(t, w - d), w + d)

    with np.errstate(all="ignore"):
        xp, zp = np.fmax(x, 1e-6), np.fmax(z, 1e-6)
        a = move(0.5 / zp, xp, 1e-4)
        b = move(0.5 / xp, zp, 1e-4)
        ex = np.where(xp < zp, a, move(0.5 / b, xp, 1e-4))
        ez = np.where(xp < zp, move(0.5 / a, zp, 1e-4), b)
    assert got[2] == 0.5
    np.testing.assert_array_equal(got[0], ex)
    np.testing.assert_array_equal(got[1], ez)
