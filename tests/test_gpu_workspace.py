"""The device workspace of one run (GPU).

A buffer of the size that a run took when its running sums had no padding and its
outputs for the host memory of their own is still enough for the run: such a size may be
a constant in a program, or a share of a server's budget.  And a run in a buffer of
exactly smc_workspace_bytes, with its results on the host, in device memory or with all
ancestors, gives the same bits as in the library's own and writes nothing past it.
"""
import numpy as np
import pytest

import inputs
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu

# bytes: FP64 with the last ancestors, FP32 with all of them (50 observations, 16 tips,
# 28 days)
ENOUGH = [
    ("lg", 1, 7680, 7680), ("lg", 1000, 71424, 255232), ("lg", 5000, 331264, 1251328),
    ("lg", 23171, 1499136, 5762560), ("lg", 46000, 2978816, 11442688),
    ("crbd", 1000, 110848, 202752), ("crbd", 23171, 2425600, 4557312),
    ("rateshift", 1000, 586496, 526848), ("rateshift", 46000, 26713600, 23953920),
    ("crbd_ds", 5000, 690432, 1110528), ("crbd_ds", 23171, 3166976, 5113344),
    ("seir", 1000, 299264, 355072), ("seir", 46000, 13466368, 16042752),
]


def _model(kind):
    if kind == "lg":
        return smc.Model("lg", obs=inputs.lg_observations(50, seed=1))
    if kind == "seir":
        return smc.Model("seir", obs=inputs.seir_observations(28, seed=3))
    tree = inputs.yule_tree(16, seed=2)
    if kind == "rateshift":
        return smc.Model("rateshift", tree=tree, sigma=0.3, lam_stack_cap=20)
    return smc.Model(kind, tree=tree)


@pytest.mark.parametrize("kind,N,last,every", ENOUGH)
def test_former_sizes_are_enough(kind, N, last, every):
    m = _model(kind)
    assert m.workspace_bytes(N, "fp64") <= last
    assert m.workspace_bytes(N, "fp32", 0, True) <= every
    m.close()


@pytest.mark.parametrize("where,every", [("host", False), ("host", True), ("device", False)])
@pytest.mark.parametrize("kind,N", [("lg", 1), ("lg", 700), ("lg", 17001), ("lg", 100001),
                                    ("rateshift", 700), ("rateshift", 5000), ("crbd", 1500)])
def test_nothing_past_the_workspace(kind, N, where, every):
    import torch

    m = _model(kind)
    need = m.workspace_bytes(N, "fp64", 0, every)
    buf = torch.full((need + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    kw = dict(where=where, record_all_ancestors=every)
    a = smc.run(m, N, 3, workspace=buf[:need], **kw)
    b = smc.run(m, N, 3, **kw)
    with pytest.raises(smc.SmcError):
        smc.run(m, N, 3, workspace=buf[:need - 1], **kw)
    torch.cuda.synchronize()
    m.close()
    assert torch.all(buf[need:] == 0x5A)
    for key in ("log_z", "final_logw", "ancestors", "real_fields", "int_fields", "stack", "resampled"):
        if key in b:
            x, y = (v.cpu().numpy() if where == "device" else v for v in (a[key], b[key]))
            np.testing.assert_array_equal(x, y, err_msg=key)
