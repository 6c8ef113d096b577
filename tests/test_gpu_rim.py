"""Pairs within rounding of the cutoff: which the gather force adds and which hacc_count_pairs counts.

With the grid-force polynomial zero the force ends at r_c with a step of
r_c (r_c^2 + eps)^-3/2 instead of vanishing there, so a pair lost by the hit
path's filter, or decided differently by the count, shows at full size."""

import numpy as np
import pytest

from gpu_util import need_cuda

pytestmark = pytest.mark.gpu

NO_POLY = np.zeros(6, np.float32)


def unit_vectors(rng, n):
    u = rng.normal(size=(n, 3))
    return u / np.linalg.norm(u, axis=1)[:, None]


def accepted_sum(sr, m, L, rc, eps, dense=None, chunk=256):
    """float64 force of the pairs that the float32 test on the binned offsets accepts (sorted order), and their number.
    An image offset is added to the j offset, or for the i of dense cells (a flag per cell) taken from the i offset."""
    o = sr.sorted4.cpu().numpy()[:, :3]
    perm = sr.perm.cpu().numpy()
    cell = sr.cell_of.cpu().numpy()[perm].astype(np.int64)
    n = round(sr.n_cells ** (1 / 3))
    w = np.float32(np.float32(L) / np.float32(n))
    xyz = np.stack([cell % n, cell // n % n, cell // (n * n)], 1)
    centre = ((xyz.astype(np.float32) + np.float32(0.5)) * w).astype(np.float64)
    L32 = float(np.float32(L))
    rc2e = np.float32(float(np.float32(rc)) ** 2 + float(np.float32(eps)))
    F, total = np.zeros((len(o), 3)), 0
    for b in range(0, len(o), chunk):
        i = slice(b, b + chunk)
        d = centre[None] - centre[i, None]
        D = (d - L32 * np.round(d / L32)).astype(np.float32)
        dx = (o[None] + D) - o[i, None]
        if dense is not None:
            dx = np.where(dense[cell[i]][:, None, None], o[None] - (o[i, None] - D), dx)
        se = np.float32(eps) * np.ones(dx.shape[:2], np.float32)
        for k in range(3):  # fmaf: the product is exact in float64
            se = (dx[..., k].astype(np.float64) ** 2 + se).astype(np.float32)
        ok = se < rc2e
        ok[np.arange(ok.shape[0]), np.arange(b, b + ok.shape[0])] = False
        t = np.where(ok, se.astype(np.float64), 1.0) ** -1.5 * ok * m[perm][None]
        F[i] = (t[..., None] * dx).sum(1)
        total += int(ok.sum())
    return F, total, perm


def planted(rng, base, L, k, rc, n):
    """About n points within a few units in the last place of r_c of a base particle (a lattice of k^3), none close to
    any other: a close pair's rounding would hide a rim term."""
    src = base[rng.integers(0, len(base), n)]
    new = src + rc * (1 + rng.integers(-8, 9, (n, 1)) * 2.0 ** -23) * unit_vectors(rng, n)
    d = new[:, None] - base[None]
    d -= L * np.round(d / L)
    return new[np.linalg.norm(d, axis=2).min(1) > 0.25 * L / k]


@pytest.mark.parametrize("rc,eps,cell,fill,plant",
                         [(3.0, 0.01, 1.0, 8, 4), (3.0, 0.01, 1.0, 26, 4), (3.0, 1e-6, 1.0, 8, 4), (3.0, 1e-6, 1.0, 26, 4),
                          (1.7, 0.3, 1.0, 26, 4), (0.05, 1e-5, 1.0, 26, 4), (40.0, 1.0, 1.0, 8, 4), (3.0, 0.01, 1.33, 20, 4),
                          (3.0, 0.01, 0.5, 4, 2), (3.0, 0.01, 0.5, 20, 4), (3.0, 0.01, 0.34, 1, 1)])
def test_no_pair_is_lost_at_the_rim(rc, eps, cell, fill, plant):
    """Cells of width `cell` r_c with about fill particles each on a jittered lattice, and plant more per cell within a
    few units in the last place of r_c of another: one or two lanes a particle, lists of up to three cells' reach,
    several softenings and scales.  (A fine mesh of many particles has too many candidates for the gather call's hit
    path; the symmetric call still takes it.)"""
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    side = 6 if cell >= 1 else 7
    L = float(np.float32(1.003 * side * cell * rc))
    rng = np.random.default_rng(fill + side)
    k = round((fill * side ** 3) ** (1 / 3))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    base = (g + 0.5 + rng.uniform(-0.15, 0.15, g.shape)) * (L / k)
    new = planted(rng, base, L, k, rc, plant * side ** 3)
    pos = (np.concatenate([base, new]) % L).astype(np.float32)
    N = len(pos)
    m = rng.uniform(0.5, 1.0, N).astype(np.float32)
    sr = hs.ShortRange(L, np.array([0, N]), rc, cell_min=cell * rc)
    prm = hs.SRParams(eps, rc, NO_POLY)
    sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(m, device="cuda"))
    count = (sr.cell_start[1:] - sr.cell_start[:-1]).cpu().numpy()
    assert count.max() <= 40 and round(sr.n_cells ** (1 / 3)) == side
    off, nbr = sr.nbr_off.cpu().numpy(), sr.nbr_cell.cpu().numpy()
    gather_hits = np.add.reduceat(count[nbr], off[:-1]).max() <= 27 * 40
    assert gather_hits or (cell, fill) == (0.5, 20)
    f, s = sr.force(prm), sr.force_symmetric(prm)
    sr.check_status()
    F, total, perm = accepted_sum(sr, m, L, rc, eps)
    rim = 0.5 * rc * (rc * rc + eps) ** -1.5  # the least that a lost pair can take away
    for name, t in (("gather", f), ("symmetric", s)):
        err = np.abs(t.cpu().numpy().T[perm] - F).max()
        assert err < 0.05 * rim or (name == "gather" and not gather_hits), (name, err, rim)
    assert sr.pairs_within_cutoff(prm) == total or not gather_hits


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_the_count_is_the_gather_force_s_own(seed):
    """Cells of the hit path beside dense ones (more than 40 particles, or a neighbourhood of more than 27 times that),
    2,600 pairs planted at the rim: the count decides each ordered pair in the form that the force uses for its i."""
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    rc, eps, side = 3.0, 0.01, 6
    L = float(np.float32(1.003 * side * rc))
    rng = np.random.default_rng(seed)
    k = 15
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    base = (g + 0.5 + rng.uniform(-0.15, 0.15, g.shape)) * (L / k)
    heavy = rng.choice(side ** 3, 40, replace=False)  # 30 more in each of these cells
    at = np.repeat(np.stack([heavy % side, heavy // side % side, heavy // side ** 2], 1), 30, axis=0)
    base = np.concatenate([base, (at + rng.uniform(0.0, 1.0, at.shape)) * (L / side)])
    pos = (np.concatenate([base, planted(rng, base, L, 4 * k, rc, 2600)]) % L).astype(np.float32)
    N = len(pos)
    m = rng.uniform(0.5, 1.0, N).astype(np.float32)
    sr = hs.ShortRange(L, np.array([0, N]), rc)
    prm = hs.SRParams(eps, rc, NO_POLY)
    sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(m, device="cuda"))
    sr.force(prm)
    sr.check_status()
    count = (sr.cell_start[1:] - sr.cell_start[:-1]).cpu().numpy()
    reach = np.add.reduceat(count[sr.nbr_cell.cpu().numpy()], sr.nbr_off.cpu().numpy()[:-1])
    dense = (count > 40) | (reach > 27 * 40)
    assert 0.1 < dense.mean() < 0.9
    _, total, _ = accepted_sum(sr, m, L, rc, eps, dense)
    assert sr.pairs_within_cutoff(prm) == total
