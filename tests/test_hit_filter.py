"""The tensor-core filter of the hit path loses no pair inside the cutoff.

The filter keeps a pair when n_i + n_j - 2 x_i.x_j - cut is negative, with
n = (1 - delta) |x|^2 and x, n_j rounded to tf32 (11 significant bits).  This
restates it in numpy with the sources' own delta and cut (the kernel itself is
held to the exact test in test_gpu_rim.py), with the products' sum truncated to float32 after every
term, on pairs at and just inside the cutoff over the offsets that cells of
one to eight cutoffs produce, and on uniform pairs, of which it may admit only
few more than the exact test."""

import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1211_4864_gb300", "csrc")


def source(name, pattern):
    """The one match of pattern in a CUDA source."""
    with open(os.path.join(CSRC, name)) as f:
        found = re.findall(pattern, f.read())
    assert len(found) == 1, (name, pattern, found)
    return found[0]


# the margin and the cut as the sources form them (hit_cut: r_c^2 (1.0 + 1.0 / A) + eps / (1 << B))
RC, EPS = np.float32(3.0), np.float32(0.01)
DELTA = np.float32(source("hacc_hits.cuh", r"constexpr float HITS_DELTA = ([0-9.e-]+)f;"))
A, B = source("hacc_pairs.cuh", r"K\.hit_cut = \(float\)\(\(double\)p->rcut \* \(double\)p->rcut \* "
                                r"\(1\.0 \+ 1\.0 / (\d+)\) \+ \(double\)p->eps / \(1 << (\d+)\)\);")
CUT = np.float32(9.0 * (1 + 1 / int(A)) + float(EPS) / 2 ** int(B))


def tf32(x):
    b = np.asarray(x, np.float32).view(np.uint32).astype(np.uint64)
    return ((b + 0x1000) & 0xFFFFE000).astype(np.uint32).view(np.float32)  # round to nearest, ties away


def trunc32(x):
    """float64 to float32 towards zero."""
    y = x.astype(np.float32)
    over = np.abs(y.astype(np.float64)) > np.abs(x)
    return np.where(over, np.nextafter(y, np.float32(0)), y)


def norm(x):
    return (x[:, 2] * x[:, 2] + (x[:, 1] * x[:, 1] + x[:, 0] * x[:, 0])).astype(np.float32)


def admitted(xi, xj):
    ni = norm(xi) * (1 - DELTA) - CUT
    nj = norm(xj) * (1 - DELTA)
    hi = tf32(ni)
    terms = [tf32(-2 * xi[:, k]).astype(np.float64) * tf32(xj[:, k]) for k in range(3)]
    terms += [tf32(nj).astype(np.float64), hi.astype(np.float64), tf32(ni - hi).astype(np.float64)]
    s = np.zeros(len(xi), np.float32)
    for t in terms:
        s = trunc32(s.astype(np.float64) + t)
    return s < 0


def inside(xi, xj):
    d = xj - xi
    se = (d[:, 2] * d[:, 2] + (d[:, 1] * d[:, 1] + (d[:, 0] * d[:, 0] + EPS))).astype(np.float32)
    return se < np.float32(9.0 + float(EPS))


@pytest.mark.parametrize("w", [1.5, 3.0, 3.9, 6.0, 12.0, 24.0])
def test_filter_keeps_every_pair_inside_the_cutoff(w):
    rng = np.random.default_rng(int(10 * w))
    n = 400000
    xi = rng.uniform(-w / 2, w / 2, (n, 3)).astype(np.float32)
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    r = np.where(rng.random(n) < 0.7, 3.0 * (1 - 10.0 ** rng.uniform(-8, -3, n)), 3.0 * rng.random(n) ** (1 / 3))
    xj = (xi + r[:, None] * u).astype(np.float32)
    ok = inside(xi, xj)
    assert ok.sum() > n // 2
    assert np.all(admitted(xi, xj)[ok])


def test_filter_admits_few_pairs_beyond_the_cutoff():
    rng = np.random.default_rng(1)
    xi = rng.uniform(-1.5, 1.5, (2000000, 3)).astype(np.float32)
    xj = rng.uniform(-4.5, 4.5, (2000000, 3)).astype(np.float32)
    kept, exact = admitted(xi, xj), inside(xi, xj)
    assert np.all(kept[exact])
    assert kept.sum() < 1.03 * exact.sum()
