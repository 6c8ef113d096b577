"""The hit path of the pair kernels (chaining-mesh cells of few particles).

Cells of n particles each at the edges of its row tiles (8, 16, 32), of the
cell size it takes (40 and 41) and of its batches of 256 candidates (27 cells
of 9 and 10, a last step of one record), small cells around one large cell
(both kernels add to the same particles; the largest is cut into segments),
and a fine mesh whose lists span
several groups of 32 entries.  Every pair call on both mass paths against the
float64 oracle; the gather calls again bit for bit."""

import numpy as np
import pytest

import oracle
from gpu_util import MAX_TOL, RMS_TOL, err_norms, need_cuda
from synth import default_coeffs

pytestmark = pytest.mark.gpu

EPS, RC = 0.01, 3.0


def cells(n, side, big=0, seed=0, L=None):
    """n particles in every cell of width 3 (side^3 of them), big more in one."""
    rng = np.random.default_rng(seed)
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)
    own = np.repeat(g, n, axis=0)
    own = np.concatenate([own, np.tile(g[len(g) // 2], (big, 1))])
    pos = (own + rng.uniform(0.001, 0.999, own.shape)) * 3.0
    return pos[rng.permutation(len(pos))].astype(np.float32), 3.0 * side


def rounding_bounds(pos, m, lam, L):
    """Per particle, what the rounding of its pairs' terms can add to a force and to a gradient component.  With t =
    (s + eps)^-1/2 from a root within two units in the last place, t^3 is off by 2^-21 of itself and a Horner sum of
    terms whose magnitudes add to at most 6 (value) or 8 (slope times s) by 6 2^-24 of them; the offsets, below 8 in
    magnitude, add 2^-22 to a distance.  The third bound is for dL/dm."""
    d = pos[None] - pos[:, None]
    d -= L * np.round(d / L)
    s = (d * d).sum(-1)
    t = (s + EPS) ** -0.5
    near = (s < RC * RC) & (s > 0)
    f = 2.0 ** -21 * (t ** 3 + 6) * np.sqrt(s) + 2.0 ** -22 * 4 * (t ** 3 + 1)
    slope = 2.0 ** -21 * (8 * t ** 3 + 16) + 2.0 ** -22 * 16 * (t ** 4 + 1)
    l = np.linalg.norm(lam, axis=1)
    mu = m[:, None] * l[None] + m[None] * l[:, None]
    return (near * m[None] * f).sum(1), (near * mu * slope).sum(1), (near * f * l[None]).sum(1)


CASES = [(1, 3, 0, 3.0, 32), (8, 3, 0, 3.0, 32), (9, 3, 0, 3.0, 32), (10, 4, 0, 3.0, 64), (16, 3, 0, 3.0, 32),
         (17, 3, 0, 3.0, 32), (32, 3, 0, 3.0, 32), (33, 3, 0, 3.0, 32), (33, 3, 0, 3.0, 64), (64, 3, 0, 3.0, 128),
         (65, 3, 0, 3.0, 128), (40, 3, 0, 3.0, 64), (41, 3, 0, 3.0, 64), (12, 3, 300, 3.0, 128), (20, 3, 70, 3.0, 32), (12, 3, 2000, 3.0, 128), (19, 4, 0, 1.5, 32), (3, 3, 0, 0.75, 32)]


@pytest.mark.parametrize("n,side,big,cell_min,split_T", CASES)
@pytest.mark.parametrize("masses", ["equal", "varied"])
def test_cells_of_every_size(n, side, big, cell_min, split_T, masses):
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    pos, L = cells(n, side, big, seed=n + big)
    N = len(pos)
    rng = np.random.default_rng(5)
    m = rng.uniform(0.5, 2.0, N).astype(np.float32) if masses == "varied" else np.full(N, 0.37, np.float32)
    lam = rng.normal(size=(N, 3)).astype(np.float32)
    c = default_coeffs(RC, EPS)
    prm = hs.SRParams(EPS, RC, c)
    sr = hs.ShortRange(L, np.array([0, N]), RC, cell_min=cell_min, split_T=split_T)
    p = torch.tensor(pos.T.copy(), device="cuda")
    lt = torch.tensor(lam.T.copy(), device="cuda")
    sr.prepare(p, torch.tensor(m, device="cuda"))
    a, phi = sr.force(prm), sr.potential(prm)
    g, gm = sr.adjoint(prm, lt)
    got = {"force": a, "symmetric": sr.force_symmetric(prm), "adjoint": g, "adjoint w": sr.adjoint(prm, lt, want_gm=False)[0]}
    gs, gms = sr.adjoint_symmetric(prm, lt)
    got["adjoint symmetric"] = gs
    got["adjoint symmetric w"] = sr.adjoint_symmetric(prm, lt, want_gm=False)[0]
    again = sr.force(prm)
    torch.cuda.synchronize()
    sr.check_status()
    c64 = c.astype(np.float64)
    A = oracle.sr_force(*pos.T.copy(), m, L, EPS, RC, c64)
    G, GM = oracle.sr_force_adjoint(*pos.T.copy(), m, L, EPS, RC, c64, lam.astype(np.float64))
    P = oracle.sr_potential(*pos.T.copy(), m, L, EPS, RC, c64)
    if n < 8:  # few pairs, most of them where f = t^3 - poly nearly cancels: the terms' own rounding
        bf, bg, bm = rounding_bounds(pos.astype(np.float64), m, lam, L)
        for name, t in got.items():
            err = np.abs(t.cpu().numpy().T - (G if "adjoint" in name else A)).max(1)
            assert np.all(err <= (bg if "adjoint" in name else bf) + 1e-9), name
        for name, t in (("adjoint gm", gm), ("adjoint symmetric gm", gms)):
            assert np.all(np.abs(t.cpu().numpy() - GM) <= bm + 1e-9), name
    else:
        for name, t in got.items():
            rms, mx = err_norms(t.cpu().numpy().T.astype(np.float64), G if "adjoint" in name else A)
            assert rms < RMS_TOL and mx < MAX_TOL, (name, rms, mx)
        for name, t in (("adjoint gm", gm), ("adjoint symmetric gm", gms)):
            rms = np.linalg.norm(t.cpu().numpy() - GM) / np.linalg.norm(GM)
            assert rms < RMS_TOL, (name, rms)
    # V = poly(se) - se^-1/2: eight Horner steps of terms below 1.5 and a root within two units in the last
    # place, so a pair is off by at most 8 2^-24 1.5 + 2^-22 (|V| + 1.5)
    bound = (8 * 1.5 * 2.0 ** -24 + 1.5 * 2.0 ** -22) * m.sum() + 2.0 ** -22 * np.abs(P)
    assert np.all(np.abs(phi.cpu().numpy() - P) < bound), "potential"
    if n >= 8:
        assert np.linalg.norm(phi.cpu().numpy() - P) / np.linalg.norm(P) < RMS_TOL
    assert torch.equal(a, again)


@pytest.mark.parametrize("what", ["tasks dropped", "wait runs out"])
def test_outputs_of_tasks_that_did_not_run_are_zero(what):
    """Small cells only: every output of a symmetric call is written, 0 where a task was dropped (and flagged)."""
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    pos, L = cells(9, 5, seed=2)
    N = len(pos)
    sr = hs.ShortRange(L, np.array([0, N]), RC)
    prm = hs.SRParams(EPS, RC, default_coeffs(RC, EPS))
    lam = torch.ones(3, N, device="cuda")
    if what == "tasks dropped":
        sr.lists.task_cap = 5
    sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.ones(N, device="cuda"))
    torch.cuda.synchronize()
    sr.status.zero_()
    launch = hs.Launch(wait_cycles=1) if what == "wait runs out" else None
    outs = [torch.full((3, N), float("nan"), device="cuda") for _ in range(2)]
    sr.force_symmetric(prm, outs[0], launch=launch)
    sr.adjoint_symmetric(prm, lam, outs[1], launch=launch)
    torch.cuda.synchronize()
    done = 45 if what == "tasks dropped" else 0  # five tasks of one cell's nine particles
    for out in outs:
        o = out.cpu().numpy()
        assert np.all(np.isfinite(o))
        assert np.count_nonzero(np.any(o != 0, axis=0)) <= done


@pytest.mark.parametrize("masses", ["equal", "varied"])
def test_stored_and_converted_totals_are_the_same_numbers(masses):
    """A symmetric call's outputs for small cells do not depend on whether a dense cell elsewhere has the sums go through
    the float64 totals: the hit kernel's own stores round the same products once.  (Its product of a mass and a
    two-word sum is exact to 2^-46, so at most one value in 2^20 falls on the other side of a tie.)"""
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    small, L = cells(20, 8, seed=6)
    rng = np.random.default_rng(8)
    blob = (0.01 + 2.98 * rng.random((300, 3))).astype(np.float32)  # one cell, dense
    own = np.all(small >= 6.0, axis=1) & np.all(small < 21.0, axis=1)  # no neighbour of that cell's
    m = rng.uniform(0.5, 2.0, len(small) + 300).astype(np.float32) if masses == "varied" else np.full(len(small) + 300, 0.37, np.float32)
    lam = rng.normal(size=(3, len(small) + 300)).astype(np.float32)
    prm = hs.SRParams(EPS, RC, default_coeffs(RC, EPS))
    outs = []
    for pos in (small, np.concatenate([small, blob])):
        N = len(pos)
        sr = hs.ShortRange(L, np.array([0, N]), RC)
        sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(m[:N], device="cuda"))
        lt = torch.tensor(lam[:, :N].copy(), device="cuda")
        f = sr.force_symmetric(prm)
        g, gm = sr.adjoint_symmetric(prm, lt)
        w, _ = sr.adjoint_symmetric(prm, lt, want_gm=False)
        torch.cuda.synchronize()
        sr.check_status()
        outs.append([t.cpu().numpy()[..., : len(small)][..., own] for t in (f, g, gm, w)])
    for a, b in zip(*outs):
        assert np.count_nonzero(a != b) <= 1 and np.allclose(a, b, rtol=2.0 ** -23, atol=0)


def fine_mesh():
    """Cells of half the cutoff (lists of up to 125 entries, four groups of 32): ten particles in each of 10^3, 3,003 in
    two that are each other's neighbours and 50 in another, so that dense tasks skip large cells and meet small ones
    before their own, over several groups."""
    rng = np.random.default_rng(12)
    g = np.stack(np.meshgrid(*[np.arange(10)] * 3, indexing="ij"), -1).reshape(-1, 3)
    n = np.full(1000, 10)
    n[[444, 556]] = 3003
    n[455] = 50
    return (np.repeat(g, n, axis=0) + rng.uniform(0.01, 0.99, (n.sum(), 3))) * 1.5, 15.0, 1.5


def crowded_cell():
    """33,283 particles in one cell: its last task holds 3, and one particle of the next cells meets more than 32,768 j
    records, so that a segment is a multiple of the usual length."""
    rng = np.random.default_rng(13)
    pos = np.concatenate([rng.uniform(3.001, 5.999, (128 * 260 + 3, 3)), rng.uniform(0.0, 9.0, (300, 3))])
    out = np.all((pos[-300:] > 3.0) & (pos[-300:] < 6.0), axis=1)
    return np.delete(pos, len(pos) - 300 + np.nonzero(out)[0], axis=0), 9.0, 3.0


@pytest.mark.parametrize("field", [fine_mesh, crowded_cell])
@pytest.mark.parametrize("masses", ["equal", "varied"])
def test_segments_of_long_lists_and_full_cells(field, masses):
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    pos, L, cell_min = field()
    rng = np.random.default_rng(14)
    pos = pos[rng.permutation(len(pos))].astype(np.float32)
    N = len(pos)
    m = rng.uniform(0.5, 2.0, N).astype(np.float32) if masses == "varied" else np.full(N, 0.37, np.float32)
    lam = rng.normal(size=(N, 3)).astype(np.float32)
    c = default_coeffs(RC, EPS)
    prm = hs.SRParams(EPS, RC, c)
    sr = hs.ShortRange(L, np.array([0, N]), RC, cell_min=cell_min, split_T=128)
    sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(m, device="cuda"))
    lt = torch.tensor(lam.T.copy(), device="cuda")
    a = sr.force_symmetric(prm)
    g, gm = sr.adjoint_symmetric(prm, lt)
    torch.cuda.synchronize()
    sr.check_status()
    start, perm = sr.cell_start.cpu().numpy(), sr.perm.cpu().numpy()
    count = np.diff(start)
    if field is fine_mesh:
        assert sr.n_entries == 1000 * 125 and count.max() > 3000
    else:
        assert count.max() > 32768 and count.max() % 128 == 3
    full = np.argsort(count)[-2:]
    tail = np.concatenate([perm[start[k + 1] - 3 : start[k + 1]] for k in full])  # the short last tasks
    t = np.unique(np.concatenate([rng.choice(N, 600, replace=False), tail, perm[start[full[1]] :][:128]]))
    c64 = c.astype(np.float64)
    A = oracle.sr_force(*pos.T.copy(), m, L, EPS, RC, c64, targets=t)
    G, GM = oracle.sr_force_adjoint(*pos.T.copy(), m, L, EPS, RC, c64, lam.astype(np.float64), targets=t)
    for name, got, ref in (("force", a, A), ("adjoint", g, G)):
        rms, mx = err_norms(got.cpu().numpy().T[t].astype(np.float64), ref)
        assert rms < RMS_TOL and mx < MAX_TOL, (name, rms, mx)
    assert np.linalg.norm(gm.cpu().numpy()[t] - GM) < RMS_TOL * np.linalg.norm(GM)


@pytest.mark.parametrize("leaf", [8, 64])
def test_segments_of_tree_lists(leaf):
    """Tree leaves about a blob of 6,000 particles: long lists whose length is estimated from sixteen entries, tasks cut
    into segments, the segments' walks starting and ending inside the list."""
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    rng = np.random.default_rng(leaf)
    pos = np.concatenate([rng.uniform(0, 18.0, (6001, 3)), 9.0 + rng.normal(size=(6000, 3))]).astype(np.float32)
    N, L = len(pos), 18.0
    m = rng.uniform(0.5, 2.0, N).astype(np.float32)
    lam = rng.normal(size=(N, 3)).astype(np.float32)
    c = default_coeffs(RC, EPS)
    prm = hs.SRParams(EPS, RC, c)
    sr = hs.ShortRange(L, np.array([0, N]), RC, builder="rcb", leaf_max=leaf, split_T=leaf)
    sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(m, device="cuda"))
    lt = torch.tensor(lam.T.copy(), device="cuda")
    a = sr.force_symmetric(prm)
    g, gm = sr.adjoint_symmetric(prm, lt)
    torch.cuda.synchronize()
    sr.check_status()
    longest = (sr.nbr_off[1 : sr.n_cells + 1] - sr.nbr_off[: sr.n_cells]).max().item()
    assert longest > 128
    t = rng.choice(N, 800, replace=False)
    c64 = c.astype(np.float64)
    A = oracle.sr_force(*pos.T.copy(), m, L, EPS, RC, c64, targets=t)
    G, GM = oracle.sr_force_adjoint(*pos.T.copy(), m, L, EPS, RC, c64, lam.astype(np.float64), targets=t)
    for name, got, ref in (("force", a, A), ("adjoint", g, G)):
        rms, mx = err_norms(got.cpu().numpy().T[t].astype(np.float64), ref)
        assert rms < RMS_TOL and mx < MAX_TOL, (name, rms, mx)
    assert np.linalg.norm(gm.cpu().numpy()[t] - GM) < RMS_TOL * np.linalg.norm(GM)
