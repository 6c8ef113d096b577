"""The order in which the pair kernels take their work.

The force calls leave their split of the task order in the workspace: four
counters (items taken and present), then, behind the cotangents and the
float64 totals, one slot a particle with the dense kernel's items from the
front and the hit kernel's tasks from the back.  Both lists keep the
heaviest-first order over several chunks of 1024 tasks; a symmetric call of up
to 2^21 particles takes the dense chunks from the last to the first."""

import numpy as np
import pytest

from gpu_util import need_cuda
from synth import default_coeffs

pytestmark = pytest.mark.gpu

CHUNK, HITS = 1024, 40


def split(sr):
    """(dense items as rows of task, segment, last; hit tasks in the order they are taken)"""
    up = lambda n: (n + 255) // 256 * 256  # noqa: E731
    ws = sr.ws.cpu().numpy()
    counts = ws[:16].view(np.int32)
    at = 256 + up(16 * sr.N) + up(32 * sr.N)
    items = ws[at : at + 8 * sr.N].view(np.int32).reshape(-1, 2)
    dense = items[: counts[2]]
    return np.stack([dense[:, 0], dense[:, 1] & 0xFFFF, dense[:, 1] >> 24], 1), items[::-1][: counts[3], 0]


@pytest.mark.parametrize("builder", ["mesh", "rcb"])
def test_the_split_keeps_the_order(builder):
    torch = need_cuda()
    import paper_1211_4864_gb300 as hs
    hs.load()
    rng = np.random.default_rng(31)
    L = 48.0
    pos = np.concatenate([rng.uniform(0, L, (60000, 3)), 24.0 + 2.5 * rng.normal(size=(40001, 3))]) % L
    N = len(pos)
    sr = hs.ShortRange(L, np.array([0, N]), 3.0, split_T=16, builder=builder, leaf_max=16)
    prm = hs.SRParams(0.01, 3.0, default_coeffs(3.0, 0.01))
    sr.prepare(torch.tensor(pos.T.astype(np.float32).copy(), device="cuda"), torch.ones(N, device="cuda"))
    nt = int(sr.n_tasks.item())
    order = sr.task_order[:nt].cpu().numpy()
    assert nt > 3 * CHUNK
    if builder == "mesh":
        count = (sr.cell_start[1:] - sr.cell_start[:-1]).cpu().numpy()
        reach = np.add.reduceat(count[sr.nbr_cell.cpu().numpy()], sr.nbr_off.cpu().numpy()[:-1])
        cell = sr.tasks[:nt, 0].cpu().numpy()[order]
        small = count[cell] <= HITS
        near = small & (reach[cell] <= 27 * HITS)
        assert near.sum() > CHUNK and (~small).sum() > CHUNK
    else:
        small = near = np.zeros(nt, bool)

    sr.force(prm)
    dense, hits = split(sr)
    assert np.array_equal(dense[:, 0], order[~near]) and np.all(dense[:, 1:] == (0, 1))
    assert np.array_equal(hits, order[near])

    sr.force_symmetric(prm)
    dense, hits = split(sr)
    assert np.array_equal(hits, order[small])
    first = dense[:, 1] == 0
    chunks = [order[c : c + CHUNK][~small[c : c + CHUNK]] for c in range(0, nt, CHUNK)]
    assert np.array_equal(dense[first, 0], np.concatenate(chunks[::-1]))
    assert np.array_equal(np.roll(dense[:, 2], 1), first)  # a task ends where the next begins
    assert np.all(np.diff(dense[:, 1])[~first[1:]] == 1) and np.all(np.diff(dense[:, 0])[~first[1:]] == 0)
    assert (~first).sum() > 0
