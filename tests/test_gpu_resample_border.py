"""Standalone resampling at the border between the calls whose CTAs combine the tile
records themselves (at most 456 tiles of 4096) and those with a combine of its own,
at the smallest sizes and with no survivor; the stack-bounded duplication at ragged
sizes (GPU)."""

import numpy as np
import pytest

import oracle
from paper_2112_00364_gb300 import smc

pytestmark = pytest.mark.gpu

TILE = 4096


@pytest.mark.parametrize("N", [1, 2, TILE, TILE + 1, 33 * TILE - 1, 455 * TILE + 1, 456 * TILE,
                               456 * TILE + 1, 457 * TILE + 13])
def test_resample_at_the_combine_border(N):
    import torch

    rng = np.random.default_rng(N)
    lw = 2.0 * rng.standard_normal(N)
    if N > 2:
        lw[rng.random(N) < 0.1] = -np.inf
    u = 0.37
    x = torch.as_tensor(lw).cuda()
    anc, out3, near = smc.resample(x, u)
    sanc, sout3, snear = smc.resample_static(x, u)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(anc.cpu().numpy(), sanc.cpu().numpy())
    np.testing.assert_array_equal(out3.cpu().numpy(), sout3.cpu().numpy())
    assert int(near) == int(snear)
    # exact ancestors from extended-precision sums; only offsets within 1e-12 N of a
    # boundary may go either way
    q = np.cumsum(np.exp(lw.astype(np.longdouble) - lw.max()))
    q *= np.longdouble(N) / q[-1]
    at = np.arange(N, dtype=np.longdouble) + np.longdouble(u)
    want = np.minimum(np.searchsorted(q, at, side="right"), N - 1)
    got = anc.cpu().numpy()
    off = np.flatnonzero(got != want)
    assert np.all(np.abs(q[np.minimum(got[off], want[off])] - at[off]) <= 1e-12 * N)
    lz = float(lw.max() + np.log(np.sum(np.exp(lw - lw.max()))) - np.log(N))
    assert abs(float(out3[2]) - lz) <= 1e-9 * max(1.0, abs(lz))


@pytest.mark.parametrize("N", [1, 5000, 456 * TILE, 456 * TILE + 1])
def test_no_survivor_at_the_combine_border(N):
    import torch

    x = torch.full((N,), -np.inf, dtype=torch.float64, device="cuda")
    near = torch.full((1,), 99, dtype=torch.int64, device="cuda")
    anc, out3, near = smc.resample(x, 0.5, n_near=near)
    np.testing.assert_array_equal(anc.cpu().numpy(), np.arange(N))
    assert out3.tolist() == [-np.inf, 0.0, -np.inf] and int(near) == 0


@pytest.mark.parametrize("N", [1, 255, 256, 1023, 1025, 4099])
@pytest.mark.parametrize("rows,bits", [(1, 32), (4, 64), (5, 32), (9, 32), (3, 64)])
def test_stack_bounded_copy(N, rows, bits):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(N + rows)
    dt = torch.float32 if bits == 32 else torch.float64
    src = torch.randn(rows, N, generator=gen, dtype=dt, device="cuda")
    dst = torch.randn(rows, N, generator=gen, dtype=dt, device="cuda")
    anc = torch.randint(0, N, (N,), generator=gen, dtype=torch.int32, device="cuda")
    sp = torch.randint(0, rows + 2, (N,), generator=gen, dtype=torch.int32, device="cuda")
    s, d, a, p = (t.cpu().numpy() for t in (src, dst, anc, sp))
    want = np.where(np.arange(rows)[:, None] < p[a][None, :], s[:, a], d)
    smc.gather(src, dst, anc, sp=sp)
    np.testing.assert_array_equal(dst.cpu().numpy(), want)
