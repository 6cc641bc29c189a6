"""Particle duplication in every form (GPU): one to nine rows of 4- and 8-byte
elements, with and without stack pointers, rows of whole and of broken 16-byte
groups, an aligned and an odd destination; against numpy, guard elements included.
"""

import numpy as np
import pytest

from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("odd", [0, 1])
@pytest.mark.parametrize("pointers", [False, True])
@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("rows", [1, 2, 3, 4, 5, 9])
@pytest.mark.parametrize("N", [1, 3, 512, 1023, 1025, 4100, 200003])
def test_every_form_of_the_copy(N, rows, bits, pointers, odd):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(N + rows)
    dt = torch.float32 if bits == 32 else torch.float64
    src = torch.randn(rows, N, generator=gen, dtype=dt, device="cuda")
    buf = torch.randn(rows * N + 8, generator=gen, dtype=dt, device="cuda")
    before = buf.cpu().numpy()
    dst = buf[odd:odd + rows * N].view(rows, N)
    anc = torch.randint(0, N, (N,), generator=gen, dtype=torch.int32, device="cuda")
    sp = None
    if pointers:
        sp = torch.randint(0, rows + 2, (N,), generator=gen, dtype=torch.int32, device="cuda")
    s, a = src.cpu().numpy(), anc.cpu().numpy()
    have = np.full(N, rows) if sp is None else sp.cpu().numpy()[a]
    old = before[odd:odd + rows * N].reshape(rows, N)
    want = before.copy()
    want[odd:odd + rows * N] = np.where(np.arange(rows)[:, None] < have[None, :], s[:, a],
                                        old).ravel()
    smc.gather(src, dst, anc, sp=sp)
    np.testing.assert_array_equal(buf.cpu().numpy(), want)
