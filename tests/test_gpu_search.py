"""The segment kernel's ancestor search on uneven populations (GPU): a few
particles that hold nearly all of the weight, so that some warps' offsets lie far
from their own tile, and others' spread over more tiles than one window holds;
beside an even population.  Weights of two values, whose exact ancestors come
from extended-precision sums; sizes at the edges of the tiles, of the runs
combined in every CTA (offsets in shared memory) and of those combined in one.
"""

import numpy as np
import pytest

import oracle
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heavy", ["few", "half"])
@pytest.mark.parametrize("N", [1025, 2047, 4097, 11000, 40001, 70001, 262145, 300001])
def test_search_on_uneven_weights(N, heavy):
    p, logw = (4.0 / N, 18.0) if heavy == "few" else (0.5, 0.4)
    seed = 3
    m = smc.Model("geometric", geo_p=p, geo_logw=logw)
    lw = smc.run(m, N, seed, max_segments=1, launch="waves")["final_logw"]
    r = smc.run(m, N, seed, max_segments=2, record_all_ancestors=True, launch="waves")
    m.close()
    assert len(np.unique(lw)) == 2
    # checkpoint 0's resampling uniform
    w = [int(v) for v in oracle.philox(np.array([[0, 0, 0, 1]]), np.array([[seed, 0]]))[0]]
    u = ((((w[1] << 32) | w[0]) >> 11) | 1) * 2.0 ** -53
    q = np.cumsum(np.exp(lw.astype(np.longdouble) - lw.max()))
    q *= np.longdouble(N) / q[-1]
    at = np.arange(N, dtype=np.longdouble) + np.longdouble(u)
    want = np.minimum(np.searchsorted(q, at, side="right"), N - 1)
    got = r["ancestors"][0]
    off = np.flatnonzero(got != want)
    # only offsets within the 1e-12 N band of a boundary may go either way
    gap = np.abs(q[np.minimum(got[off], want[off])] - at[off])
    assert np.all(gap <= 1e-12 * N), (off[:5], gap.max())
    assert np.all(np.diff(got) >= 0) and got[0] >= 0 and got[-1] < N
