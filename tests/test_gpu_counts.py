"""The Poisson and negative binomial samplers' single-precision decisions against
the oracle's FP64 samplers, draw by draw (GPU): counts and the blocks they used
are integers and must be equal, from the smallest means across the border at 10
where both change algorithm."""

import numpy as np
import pytest

import oracle
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dist,p1,p2", [
    ("poisson", 1e-300, 0), ("poisson", 1e-9, 0), ("poisson", 0.01, 0), ("poisson", 0.7, 0),
    ("poisson", 4.5, 0), ("poisson", 9.96, 0), ("poisson", 9.97, 0), ("poisson", 9.9999, 0),
    ("poisson", 10.0001, 0), ("neg_binomial", 1.0, 1e-10), ("neg_binomial", 1.0, 0.01),
    ("neg_binomial", 1.0, 9.9), ("neg_binomial", 1.0, 10.1), ("neg_binomial", 3.0, 0.5),
    ("neg_binomial", 40.0, 0.02), ("neg_binomial", 40.0, 0.2497), ("neg_binomial", 500.0, 0.0199),
    ("neg_binomial", 1000.0, 0.01)])
def test_counts_equal_the_oracles(dist, p1, p2):
    m = 400_000
    g, blocks = smc.sample(dist, m, p1, p2, seed=13)
    o, ob = oracle.sample(dist, m, p1, p2, seed=13, return_blocks=True)
    np.testing.assert_array_equal(g.cpu().numpy(), o)
    np.testing.assert_array_equal(blocks.cpu().numpy(), ob)
