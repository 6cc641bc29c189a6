"""Binomial draws of large n p (1 - p) near the centre of the rejection's triangle (GPU).

The rejection's offset x = (2a/us + b) u + n p + 1/2 moves by (4a + b) 2^-32 between
a uniform and its leading 32 bits, 1.3e-5 at n = 2e9: more than single
precision's own error there.  p is set so that the whole uniform's x lies just above
a whole number and that of its leading bits below it: the draw is the oracle's.  (Only
those draws are compared: log k! is 1e10 here, so the oracle's own acceptance test of
other candidates is rounded by 2e-6.)
"""
import math
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu

N_TRIALS = 2_000_000_000
SEED = 11


def _offset(p, u):
    b = 1.15 + 2.53 * math.sqrt(N_TRIALS * p * (1.0 - p))
    a = -0.0873 + 0.0248 * b + 0.01 * p
    x = (2 * Fraction(a) / (Fraction(1, 2) - abs(u)) + Fraction(b)) * u
    return x + N_TRIALS * Fraction(p) + Fraction(1, 2), (4.0 * a + b) * 2.0 ** -32


def _cases(count):
    """(index, p): draws whose first uniform lies within 6e-6 of 1/2."""
    m = 1 << 20
    ctr = np.zeros((m, 4), dtype=np.uint32)
    ctr[:, 0] = np.arange(m)
    w = oracle.philox(ctr, np.tile(np.array([[SEED, 0]], dtype=np.uint32), (m, 1))).astype(np.int64)
    near = np.abs(w[:, 1] - (1 << 31)) < 6e-6 * 2.0 ** 32
    # the low word counts; the second uniform accepts the candidate at once
    ok = near & (w[:, 0] > 1 << 31) & (w[:, 3] > 1 << 20) & (w[:, 3] < 0.85 * 2.0 ** 32)
    for i in np.flatnonzero(ok)[:count]:
        bits = (((int(w[i, 1]) << 32) | int(w[i, 0])) >> 11) | 1
        u = Fraction(bits, 1 << 53) - Fraction(1, 2)
        t, gap = _offset(0.3, u)
        above = Fraction(0.35 * gap * int(w[i, 0]) / 2.0 ** 32)
        yield int(i), float(Fraction(0.3) + (math.floor(t) + 1 + above - t) / N_TRIALS)


def test_draws_at_a_whole_number():
    cases = list(_cases(5))
    assert len(cases) == 5
    for i, p in cases:
        g, blocks = smc.sample("binomial", i + 1, float(N_TRIALS), p, seed=SEED)
        o, ob = oracle.sample("binomial", i + 1, float(N_TRIALS), p, seed=SEED, return_blocks=True)
        assert g[i].item() == o[i] and blocks[i].item() == ob[i] == 1, (i, p)
