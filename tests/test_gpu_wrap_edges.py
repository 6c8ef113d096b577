"""Coordinates at the edges of the wrap's short cuts, bit for bit.

The binning divides by the box side only for coordinates outside [-L, 2L)
(float64 positions: outside (0, L)) and the drift only for positions that
leave (0, L); every edge of those ranges, and values far outside, must bin and
drift as the full formula does (the oracle's, and the float64 expression)."""

import numpy as np
import pytest

import oracle
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def edges(L):
    L = np.float32(L)
    up, dn = np.float32(np.inf), np.float32(-np.inf)
    v = [0.0, -0.0, 1e-45, -1e-45, 1e-30, -1e-30, 1e-7, -1e-7, np.nextafter(L, dn), L, np.nextafter(L, up), -L,
         np.nextafter(-L, up), np.nextafter(-L, dn), 2 * L, np.nextafter(2 * L, dn), np.nextafter(2 * L, up), -2 * L,
         np.nextafter(-2 * L, up), 2.5 * L, -3.5 * L, 1000 * L, -1000.3 * L, 0.5 * L, L / 3]
    return np.array(v, np.float32)


@pytest.mark.parametrize("L", [9.0, 12.7, 16.0, 67.0])
@pytest.mark.parametrize("displaced", [False, True])
def test_binning_at_the_edges(L, displaced):
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    e = edges(L)
    x, y, z = (a.ravel().astype(np.float32) for a in np.meshgrid(e, e[::-1], e[3:9], indexing="ij"))
    N = len(x)
    m = np.ones(N, np.float32)
    d = None
    if displaced:
        d = np.random.default_rng(3).choice(np.array([0, 1e-7, -1e-7, 0.25, -0.25, L, -L], np.float32), (3, N))
    sr = hs.ShortRange(L, np.array([0, N]), 3.0)
    up = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    sr.bin(up(x), up(y), up(z), up(m), None if d is None else up(d))
    torch.cuda.synchronize()
    ref = oracle.bin_volume(x, y, z, m, L, 3.0, disp=d)
    assert np.array_equal(sr.cell_of.cpu().numpy(), ref["cell_of"])
    assert np.array_equal(sr.perm.cpu().numpy(), ref["perm"])
    assert np.array_equal(sr.sorted4.cpu().numpy(), ref["sorted4"])


@pytest.mark.parametrize("L", [9.0, 12.7, 67.0])
def test_drift_at_the_edges(L):
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    e = edges(L)
    x, v = (a.ravel().astype(np.float32) for a in np.meshgrid(e, np.array([0, 1e-9, -1e-9, 3.0, -3.0], np.float32)))
    N = len(x)
    sr = hs.ShortRange(L, np.array([0, N]), 3.0)
    pos = torch.tensor(np.stack([x, x[::-1].copy(), x]), device="cuda")
    vel = torch.tensor(np.stack([v, v[::-1].copy(), -v]), device="cuda")
    p0, v0 = pos.cpu().numpy().astype(np.float64), vel.cpu().numpy().astype(np.float64)
    h = float(np.float32(0.25))
    sr.stream(vel, pos, h)
    L64 = float(np.float32(L))
    p = p0 + h * v0
    p = p - L64 * np.floor(p / L64)
    ref = p.astype(np.float32)
    ref[ref >= np.float32(L)] = 0.0
    assert np.array_equal(pos.cpu().numpy(), ref)
