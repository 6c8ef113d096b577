"""Softenings down to the smallest normal float32 on the hit path.

A pair of a particle with itself has d = 0 and no force, but f(0) and f'(0)
grow with the softening's inverse powers: they overflow below 1e-25 (f) and
1e-15 (f'), and before that multiply the rounding of m lam - m lam.  The hit
path leaves the pair out, so every call on small cells is finite and as exact
at a tiny softening as at the usual one: on full neighbourhoods (walked by
masks) and on lone cells (every candidate inside the cutoff, walked densely),
with one and with two lanes per particle."""

import numpy as np
import pytest

import oracle
from gpu_util import err_norms, need_cuda
from synth import default_coeffs

pytestmark = pytest.mark.gpu

RC = 3.0
# Jittered unit lattice: pairs are at least 0.6 apart.  Offsets below 8 in
# magnitude add 2^-22 to a distance, 2^-22 / 0.6 of it, and the steepest term
# (f' s) carries five times that.
TOL = 5 * 2.0 ** -22 / 0.6


def particles(kind):
    rng = np.random.default_rng(17)
    g = np.stack(np.meshgrid(*[np.arange(9)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.float64)
    if kind != "full":  # the middle cell alone
        g = g[np.all((g >= 3) & (g < 6), axis=1)][: 27 if kind == "lone 27" else 12]
    return (g + 0.5 + rng.uniform(-0.2, 0.2, g.shape)).astype(np.float32)


@pytest.mark.parametrize("kind", ["full", "lone 27", "lone 12"])
@pytest.mark.parametrize("masses", ["equal", "varied"])
@pytest.mark.parametrize("eps", [2e-38, 1e-30, 1e-18, 1e-10, 1e-8, 0.01])
def test_small_cells_at_every_softening(eps, masses, kind):
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    pos = particles(kind)
    N = len(pos)
    rng = np.random.default_rng(3)
    m = rng.uniform(0.5, 2.0, N).astype(np.float32) if masses == "varied" else np.full(N, 0.37, np.float32)
    lam = rng.normal(size=(N, 3)).astype(np.float32)
    c = default_coeffs(RC, 0.01)
    prm = hs.SRParams(eps, RC, c)
    sr = hs.ShortRange(9.0, np.array([0, N]), RC)
    lt = torch.tensor(lam.T.copy(), device="cuda")
    sr.prepare(torch.tensor(pos.T.copy(), device="cuda"), torch.tensor(m, device="cuda"))
    g, gm = sr.adjoint(prm, lt)
    gs, gms = sr.adjoint_symmetric(prm, lt)
    forces = [sr.force(prm), sr.force_symmetric(prm)]
    grads = [g, gs, sr.adjoint(prm, lt, want_gm=False)[0], sr.adjoint_symmetric(prm, lt, want_gm=False)[0]]
    phi = sr.potential(prm)
    torch.cuda.synchronize()
    sr.check_status()
    e = float(np.float32(eps))
    c64 = c.astype(np.float64)
    A = oracle.sr_force(*pos.T.copy(), m, 9.0, e, RC, c64)
    G, GM = oracle.sr_force_adjoint(*pos.T.copy(), m, 9.0, e, RC, c64, lam.astype(np.float64))
    P = oracle.sr_potential(*pos.T.copy(), m, 9.0, e, RC, c64)
    for k, t in enumerate(forces):
        assert err_norms(t.cpu().numpy().T, A)[0] < TOL, ("force", k)
    for k, t in enumerate(grads):
        assert err_norms(t.cpu().numpy().T, G)[0] < TOL, ("gradient", k)
    for k, t in enumerate([gm, gms]):
        assert np.linalg.norm(t.cpu().numpy() - GM) <= TOL * np.linalg.norm(GM), ("mass gradient", k)
    assert np.linalg.norm(phi.cpu().numpy() - P) <= TOL * np.linalg.norm(P)
