"""Large sets that fill a part of their box: few nodes to a cell on average, hundreds in each occupied one."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _clusters(n, share, per_cell):
    """n nodes in `share` of the cells of a grid whose occupied cells hold about per_cell; 2 h is a cell's side."""
    rng = np.random.default_rng(n + per_cell)
    side = int(np.sqrt(n / (per_cell * share)))
    cell = rng.choice(side * side, int(share * side * side), replace=False)[rng.integers(0, int(share * side * side), n)]
    return np.stack([(cell % side + rng.random(n)) / side, (cell // side + rng.random(n)) / side], 1), np.full(n, 0.4995 / side)


def _search(xy, h, reps):
    """(row_ptr, col, best time in s of a search)"""
    import torch

    from paper_1912_06441_gb300 import Labfm

    L = Labfm(0)
    X, H = torch.from_numpy(xy).to("cuda"), torch.from_numpy(h).to("cuda")
    best = np.inf
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        L.build_neighbours(X, H, False)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e-3)
    rp, col = (t.cpu().numpy() for t in L.get_neighbours())
    L.close()
    return rp, col, best


@pytest.mark.parametrize("n,share,per_cell", [(200000, 0.05, 100), (200000, 0.02, 300), (400000, 0.3, 20), (400000, 0.1, 40)])
def test_rows_of_clustered_sets(n, share, per_cell):
    xy, h = _clusters(n, share, per_cell)
    rp, col, _ = _search(xy, h, 1)
    q = np.sort(np.random.default_rng(0).choice(n, 2000, replace=False))
    orp, ocol = oracle.neighbours_large(xy, h, False, queries=q)
    assert np.array_equal(rp[q + 1] - rp[q], np.diff(orp))
    assert np.array_equal(np.concatenate([col[rp[i]:rp[i + 1]] for i in q]), ocol)


def test_time_per_entry_of_a_clustered_set():
    """Rows of 300 against the rows of 25 of a uniform set: 1.2 times the time per entry, 7 times where each thread sorted its
    row by insertion; 3 allowed."""
    n = 200000
    rp, _, t = _search(*_clusters(n, 0.02, 300), 8)
    rng = np.random.default_rng(1)
    urp, _, ut = _search(rng.random((2 * n, 2)), np.full(2 * n, 0.5 * np.sqrt(25.0 / (2 * n * np.pi))), 8)
    assert t / rp[-1] <= 3.0 * ut / urp[-1]
