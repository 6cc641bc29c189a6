"""Negative binomial counts with parameters beyond the range of single precision
(GPU): what the single-precision decision cannot hold is drawn in FP64, as the
oracle draws it.  Shapes and rates of 2^-600 .. 2^600, ratios from below the
smallest float up, and the delayed-sampling CRBD whose priors' scales put them there.
"""
import numpy as np
import pytest

import inputs
import oracle
from paper_2112_00364_gb300 import smc
from parity import assert_parity_fp64, run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha,tau", [
    (2.0 ** 512, 2.0 ** -512), (2.0 ** 130, 2.0 ** -129), (2.0 ** 256, 2.0 ** -300),
    (2.0 ** -600, 2.0 ** 20), (2.0 ** -127, 2.0 ** 127), (1.0, 2.0 ** -130), (0.5, 2.0 ** -101),
    (2.0 ** -100, 3.0), (2.0 ** 99, 2.0 ** -99), (2.0 ** 101, 2.0 ** -100)])
def test_counts_equal_the_oracles(alpha, tau):
    m = 100_000
    g, blocks = smc.sample("neg_binomial", m, alpha, tau, seed=17)
    o, ob = oracle.sample("neg_binomial", m, alpha, tau, seed=17, return_blocks=True)
    np.testing.assert_array_equal(g.cpu().numpy(), o)
    np.testing.assert_array_equal(blocks.cpu().numpy(), ob)


@pytest.mark.parametrize("launch_n", [700, 3001])
@pytest.mark.parametrize("scale", [2.0 ** -512, 2.0 ** -130])
def test_delayed_sampling_prior_scales(scale, launch_n):
    tree = inputs.yule_tree(6, seed=5)
    g, o = run_pair("crbd_ds", launch_n, seed=4, tree=tree, lambda_scale=scale, call_limit=200)
    assert_parity_fp64(g, o)
