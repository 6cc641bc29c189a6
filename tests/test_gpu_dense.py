"""The sparse and dense forms of the segment kernel (GPU): a wave takes the dense
one above 152 x 768 = 116,736 threads.  Runs of every CTA size give the same bits
in a batch beyond that line as alone below it; one run lies a particle past it.
"""

import numpy as np
import pytest

import inputs
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu

LINE = 152 * 768


def _model(kind):
    tree = inputs.yule_tree(9, seed=21)
    if kind == "lg":
        return smc.Model(kind, obs=inputs.lg_observations(9, seed=4))
    if kind == "seir":
        return smc.Model(kind, obs=inputs.seir_observations(9, seed=7))
    if kind == "geometric":
        return smc.Model(kind)
    if kind == "rateshift":
        return smc.Model(kind, tree=tree, sigma=0.3, lam_stack_cap=tree.max_pending_right() + 1)
    return smc.Model(kind, tree=tree)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["lg", "crbd", "rateshift", "crbd_ds", "seir", "geometric"])
def test_dense_and_sparse_forms_agree(kind, precision):
    m = _model(kind)
    specs = [dict(N=n, seed=50 + q, run_id=q)
             for q, n in enumerate([LINE + 1, LINE, 30001, 9001, 4097, 300])]
    batch = smc.run_batch([m] * len(specs), specs, precision=precision)
    for sp, b in zip(specs, batch):
        a = smc.run(m, sp["N"], sp["seed"], run_id=sp["run_id"], precision=precision,
                    launch="waves")
        assert b["run_status"] == a["run_status"] and b["n_segments"] == a["n_segments"]
        assert b["log_z_value"] == a["log_z_value"]
        for name in ("final_logw", "int_fields", "real_fields"):
            if name in a:
                np.testing.assert_array_equal(b[name], a[name])
    m.close()
