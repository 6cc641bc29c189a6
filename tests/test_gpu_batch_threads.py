"""Batches of several models from many threads at once (GPU): more calls in flight than
there are idle sets of chain streams, each on a stream of its own or on the default
one, direct and captured; every result is that of the same batch called alone.
"""
import threading

import numpy as np
import pytest

import inputs
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu


def test_batches_in_flight_together():
    import torch

    tree = inputs.yule_tree(5, seed=4)
    models = [smc.Model("lg", obs=inputs.lg_observations(9, seed=1)), smc.Model("crbd", tree=tree),
              smc.Model("crbd_ds", tree=tree)]
    sizes = (700, 1500, 40, 5000)

    def specs(t):
        return ([models[(t + q) % 3] for q in range(4)],
                [dict(N=n, seed=10 * t + q, run_id=q) for q, n in enumerate(sizes)])

    def call(t, stream, graph=False):
        ms, sp = specs(t)
        return smc.run_batch(ms, sp, stream=stream, launch_graph=graph)

    alone = [call(t, None) for t in range(9)]
    wrong = []

    def work(t):
        try:
            stream = torch.cuda.Stream() if t % 3 else None
            for rep in range(6):
                for a, b in zip(alone[t], call(t, stream, graph=t % 3 == 2 and rep % 2 == 1)):
                    for key in ("log_z", "final_logw", "ancestors", "real_fields", "int_fields"):
                        np.testing.assert_array_equal(a[key], b[key], err_msg=key)
        except BaseException as e:  # noqa: BLE001 (reported by the main thread)
            wrong.append((t, repr(e)[:300]))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(9)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    for m in models:
        m.close()
    assert not wrong, wrong
