"""The resampling decision at its threshold in every launch form (GPU).

A run gives the same bits alone (cluster, one CTA, waves), in a batch and in the
server, also where the effective sample size equals the threshold to the last bits:
a population of equal weights has ESS = N, and tau = 1 compares the two.  Weights of
many values, so that the roundings of the sums differ.
"""
import numpy as np
import pytest

from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu

KEYS = ("log_z", "final_logw", "ancestors", "int_fields", "resampled", "n_resamples", "n_ess_near")


@pytest.mark.parametrize("N", [96, 320, 500, 800, 960, 1023])
def test_equal_weights_at_the_threshold(N):
    rng = np.random.Generator(np.random.PCG64(N))
    models = [smc.Model("geometric", geo_p=1.0, geo_logw=w) for w in rng.uniform(-3.0, 3.0, 40)]
    kw = dict(max_segments=2, ess_threshold=1.0)
    batch = smc.run_batch(models, [dict(N=N, seed=7, **kw)] * len(models))
    server = smc.Server(1 << 28)
    tickets = [server.submit(m, N, 7, **kw) for m in models]
    served = [server.wait(t) for t in tickets]
    server.close()
    for m, b, s in zip(models, batch, served):
        forms = [smc.run(m, N, 7, launch=f, **kw) for f in ("cluster", "one_cta", "waves")]
        m.close()
        for r in [*forms[1:], b, s]:
            for key in KEYS:
                np.testing.assert_array_equal(forms[0][key], r[key], err_msg=key)


@pytest.mark.parametrize("tau", [0.3, 0.5, 0.9, 1.0])
def test_uneven_weights_in_every_form(tau):
    """Weights whose tiles' references differ by many powers of two."""
    N = 960
    obs = np.random.Generator(np.random.PCG64(3)).normal(0.0, 20.0, 40)
    m = smc.Model("lg", obs=obs, r_sd=0.3, q_sd=4.0)
    forms = [smc.run(m, N, 9, ess_threshold=tau, record_all_ancestors=True, launch=f)
             for f in ("cluster", "one_cta", "waves")]
    forms += smc.run_batch([m], [dict(N=N, seed=9, ess_threshold=tau)], record_all_ancestors=True)
    m.close()
    for r in forms[1:]:
        for key in (*KEYS, "real_fields"):
            np.testing.assert_array_equal(forms[0][key], r[key], err_msg=key)
