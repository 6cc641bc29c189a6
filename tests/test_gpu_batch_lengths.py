"""Batches of runs of different lengths (GPU): a wave launches the CTAs of the runs
it still advances.  Every run gives the bits of the same run alone: lengths of one
and two segments, equal lengths, the longest run first, last and alone in its CTA
size, step limits below the model's length, beside a run of unknown length.
"""

import numpy as np
import pytest

import inputs
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["launches", "graph", "limits", "unknown"])
@pytest.mark.parametrize("lengths", [(1, 2, 7, 7, 40, 3), (33, 1, 1, 2, 2, 5), (4, 4, 4, 4, 4, 50)])
def test_runs_of_uneven_length(lengths, mode):
    import torch

    sizes = [700, 5000, 701, 1030, 5001, 40001]
    models = [smc.Model("lg", obs=inputs.lg_observations(t, seed=3 + t)) for t in lengths]
    specs = [dict(N=n, seed=20 + q, run_id=q) for q, n in enumerate(sizes)]
    models.append(smc.Model("crbd", tree=inputs.yule_tree(4, seed=8)))
    specs.append(dict(N=5000, seed=31, run_id=9))
    if mode == "limits":
        for q in (1, 4, 6):
            specs[q]["max_segments"] = 2
    if mode == "unknown":
        models.append(smc.Model("geometric"))
        specs.append(dict(N=900, seed=32, run_id=10))
    stream = torch.cuda.Stream() if mode == "graph" else None
    batch = smc.run_batch(models, specs, stream=stream, launch_graph=mode == "graph")
    for m, sp, b in zip(models, specs, batch):
        a = smc.run(m, sp["N"], sp["seed"], run_id=sp["run_id"], launch="waves",
                    max_segments=sp.get("max_segments", 0))
        assert b["run_status"] == a["run_status"] and b["n_segments"] == a["n_segments"]
        assert b["log_z_value"] == a["log_z_value"]
        for name in ("final_logw", "int_fields", "real_fields", "ancestors"):
            if name in a:
                np.testing.assert_array_equal(b[name], a[name])
    for m in models:
        m.close()
