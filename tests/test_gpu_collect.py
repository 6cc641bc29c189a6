"""A batch's outputs in device memory (GPU): one collecting launch for runs of very
different sizes, each with every ancestor row or the last alone.  Every output is that
of the run alone with its results on the host, and nothing is written past it.
"""
import numpy as np
import pytest

import inputs
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu

FILL = -7


def _padded(shape, dt):
    import torch

    n = int(np.prod(shape))
    buf = torch.full((n + 64,), FILL, dtype=dt, device="cuda")
    return buf, buf[:n].view(*shape)


@pytest.mark.parametrize("record_all", [False, True])
@pytest.mark.parametrize("sizes", [(1, 300001, 33), (70000,), (255, 256, 257, 8191, 8192, 8193, 1)])
def test_batch_outputs(sizes, record_all):
    import torch

    models, specs, bufs = [], [], []
    for q, n in enumerate(sizes):
        if q % 3 == 2:
            tree = inputs.yule_tree(6, seed=3 + q)
            m = smc.Model("rateshift", tree=tree, sigma=0.3, lam_stack_cap=tree.max_pending_right() + 1)
        elif q % 3 == 1:
            m = smc.Model("crbd", tree=inputs.yule_tree(8, seed=3 + q))
        else:
            m = smc.Model("lg", obs=inputs.lg_observations(14, seed=3 + q))
        rows = m.n_segments - 1 if record_all else 1
        f8, i4 = torch.float64, torch.int32
        shapes = dict(log_z=((1,), f8), final_logw=((n,), f8), ancestors=((rows, n), i4),
                      real_fields=((m.n_real, n), f8), int_fields=((m.n_int, n), i4),
                      resampled=((rows,), i4))
        if m.stack_cap:
            shapes["stack"] = ((m.stack_cap, n), f8)
        both = {k: _padded(s, dt) for k, (s, dt) in shapes.items()}
        models.append(m)
        bufs.append({k: b for k, (b, _) in both.items()})
        specs.append(dict(N=n, seed=40 + q, run_id=q, outputs={k: v for k, (_, v) in both.items()}))
    batch = smc.run_batch(models, specs, where="device", record_all_ancestors=record_all)
    torch.cuda.synchronize()
    for m, sp, b, buf in zip(models, specs, batch, bufs):
        a = smc.run(m, sp["N"], sp["seed"], run_id=sp["run_id"], launch="waves",
                    record_all_ancestors=record_all)
        m.close()
        for key, whole in buf.items():
            np.testing.assert_array_equal(b[key].cpu().numpy(), a[key], err_msg=key)
            assert torch.all(whole[-64:] == FILL), key
