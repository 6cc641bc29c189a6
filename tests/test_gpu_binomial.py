"""The binomial sampler's single-precision decisions against the oracle's FP64
sampler, draw by draw (GPU): both algorithms (inversion below mean 10, rejection
from there) around their border, small and large counts, p on both sides of 1/2
and at its ends.  A draw is an integer and the blocks it used are an integer:
both must be equal."""

import numpy as np
import pytest

import oracle
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [
    (1, 0.5), (1, 1e-9), (2, 0.999999), (19, 0.5), (20, 0.5), (21, 0.5), (40, 0.2499), (40, 0.25),
    (40, 0.2501), (100, 0.9), (100, 0.1), (101, 1.0 - 0.1), (7370, 1e-6), (7370, 0.00135),
    (7370, 0.00136), (7370, 0.37), (7370, 1.0 - 1e-7), (22110, 6.0 / 7.0), (22110, 1.0 / 7.0),
    (737000, 1.0 / 7.0), (737000, 6.0 / 7.0), (737000, 0.5), (737000, 1.3e-5), (737000, 1.4e-5),
    (2000000000, 3e-9), (2000000000, 0.3)])
def test_binomial_draws_equal_the_oracles(n, p):
    m = 300_000
    g, blocks = smc.sample("binomial", m, float(n), p, seed=11)
    o, ob = oracle.sample("binomial", m, float(n), p, seed=11, return_blocks=True)
    np.testing.assert_array_equal(g.cpu().numpy(), o)
    np.testing.assert_array_equal(blocks.cpu().numpy(), ob)
