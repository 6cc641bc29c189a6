"""A linear-Gaussian population resumed at its first block (GPU, against the oracle).

The snapshot's int field is the block that a particle goes on with.  A program that
starts a filter from particles of its own at a later observation may set it to
block 0, which draws x0 anew, then block 1 draws the step: in that order from the
particle's stream, whatever the launch form draws ahead of the checkpoint.
"""
import numpy as np
import pytest

import inputs
import oracle
from paper_2112_00364_gb300 import smc
from parity import assert_parity_exact, assert_parity_fp64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [200, 900, 30000, 100000])
def test_population_at_block_zero(N, precision):
    p = dict(obs=inputs.lg_observations(12, seed=2))
    prec = oracle.FP64 if precision == "fp64" else oracle.FP32
    m = smc.Model("lg", **p)
    snap = smc.run(m, N, 3, precision=precision, max_segments=4)
    ints = np.array(snap["int_fields"])
    ints[0, ::3] = 0
    snap = dict(snap, int_fields=ints)
    g = smc.run(m, N, 3, precision=precision, record_all_ancestors=True, resume_from=snap)
    m.close()
    o = oracle.smc_run("lg", N, 3, precision=prec, resume_from=snap, follow=g["ancestors"],
                       record_ancestors=True, **p)
    (assert_parity_fp64 if precision == "fp64" else assert_parity_exact)(g, o)


@pytest.mark.parametrize("N", [900, 100000])
def test_draws_are_counted_where_a_block_ran(N):
    """No resampling, so every particle's blocks are known: a stopped one draws nothing."""
    T, k = 12, 4
    kw = dict(ess_threshold=1e-12)
    m = smc.Model("lg", obs=inputs.lg_observations(T, seed=2))
    snap = smc.run(m, N, 3, max_segments=k, **kw)
    ints = np.array(snap["int_fields"])
    ints[0, ::3] = 0
    ints[0, 1::3] = -1
    g = smc.run(m, N, 3, resume_from=dict(snap, int_fields=ints), **kw)
    m.close()
    assert g["n_resamples"] == 0
    fresh, stopped = len(ints[0, ::3]), len(ints[0, 1::3])
    assert g["n_draws"] == (N - stopped) * (T - k) + fresh
