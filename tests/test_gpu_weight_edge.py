"""Log-weights at their tile's power-of-two reference (GPU, against the oracle).

A weight is formed relative to 2^k with k = ceil(M / ln 2), M the largest
log-weight.  Where M is log(2^k) itself, or a running sum of such values, that
quotient is rounded onto the integer k although M may lie above k ln 2 by the
rounding of M: the particle's weight is 1 there.  The geometric program's log-weight
takes these values, in every launch form; a program whose particles all carry
such a weight (geo_p = 1), one where the others weigh 1 (geo_p = 1/2), and
log-weights that accumulate because no checkpoint resamples.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2112_00364_gb300 import smc
from parity import assert_parity_exact, assert_parity_fp64

pytestmark = pytest.mark.gpu

EXPONENTS = [k for k in range(-16, 25) if k]
SEGMENTS = 3


def _oracle(g, N, precision, p, logw, segments, ess):
    return oracle.smc_run("geometric", N, 5, max_segments=segments, follow=g["ancestors"],
                          precision=oracle.FP64 if precision == "fp64" else oracle.FP32,
                          record_ancestors=True, ess_threshold=ess,
                          follow_resampled=g["resampled"] if ess else None, geo_p=p, geo_logw=logw)


def _compare(g, N, precision, p, logw, segments=SEGMENTS, ess=0.0):
    o = _oracle(g, N, precision, p, logw, segments, ess)
    assert np.isfinite(o["log_z"])
    (assert_parity_fp64 if precision == "fp64" else assert_parity_exact)(g, o)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("launch,N", [("cluster", 1000), ("one_cta", 1000), ("waves", 1000),
                                      ("waves", 20011)])
@pytest.mark.parametrize("p", [0.5, 1.0])
def test_power_of_two_weights(p, launch, N, precision):
    for k in EXPONENTS:
        logw = math.log(2.0 ** k)
        m = smc.Model("geometric", geo_p=p, geo_logw=logw)
        g = smc.run(m, N, 5, max_segments=SEGMENTS, record_all_ancestors=True, launch=launch,
                    precision=precision)
        m.close()
        _compare(g, N, precision, p, logw)


@pytest.mark.parametrize("p", [0.5, 1.0])
def test_power_of_two_weights_in_a_batch(p):
    N = 700
    models = [smc.Model("geometric", geo_p=p, geo_logw=math.log(2.0 ** k)) for k in EXPONENTS]
    got = smc.run_batch(models, [dict(N=N, seed=5, max_segments=SEGMENTS)] * len(models),
                        record_all_ancestors=True)
    for m, k, g in zip(models, EXPONENTS, got):
        m.close()
        _compare(g, N, "fp64", p, math.log(2.0 ** k))


@pytest.mark.parametrize("launch", ["cluster", "waves"])
@pytest.mark.parametrize("factor", [0.5, 2.0, 1.0 / 16.0])
def test_accumulated_power_of_two_weights(factor, launch):
    """Equal weights never fall below the threshold: 60 checkpoints' log-weights add up."""
    N, segments, logw = 900, 60, math.log(factor)
    m = smc.Model("geometric", geo_p=1.0, geo_logw=logw)
    g = smc.run(m, N, 5, max_segments=segments, record_all_ancestors=True, launch=launch,
                ess_threshold=0.5)
    m.close()
    assert g["n_resamples"] == 0
    assert abs(g["log_z_value"] - segments * logw) <= 1e-9 * abs(segments * logw)
    _compare(g, N, "fp64", 1.0, logw, segments, 0.5)
