"""Stencil rows against the oracle's all-pairs search, index by index: rows around 32, 64 and 128 entries and longer
ones (each sorted another way), boxes of one to four cells a side with and without wrap-around, and row
offsets of one block of the prefix sum, of several, and of more than it adds up directly."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _search(xy, h, periodic):
    import torch

    from paper_1912_06441_gb300 import Labfm

    dev = torch.device("cuda", 0)
    L = Labfm(0)
    L.build_neighbours(torch.from_numpy(xy).to(dev), torch.from_numpy(h).to(dev), periodic)
    rp, col = L.get_neighbours()
    got = rp.cpu().numpy(), col.cpu().numpy()
    L.close()
    return got


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n,radius", [(1, 0.1), (700, 0.3), (2047, 0.06), (2048, 0.11), (2049, 0.24), (4097, 0.05),
                                      (1500, 0.4), (900, 0.7)])
def test_rows_of_every_length(n, radius, periodic):
    """2 h_i between 0.3 and 1 of `radius`: rows of a few to hundreds of entries in one set, 1 to 20 cells a side."""
    rng = np.random.default_rng(n)
    xy = rng.random((n, 2))
    h = 0.5 * radius * (0.3 + 0.7 * rng.random(n))
    rp, col = _search(xy, h, periodic)
    orp, ocol = oracle.neighbours(xy, h, periodic)
    assert np.array_equal(rp, orp) and np.array_equal(col, ocol)


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n,spacings", [(200000, 2.3), (200001, 2.6), (400000, 2.9), (399999, 2.9)])
def test_large_sets_of_few_nodes_a_cell(n, spacings, periodic):
    """Random nodes around the sizes where the search changes its sweep, 5 to 8 nodes a cell on average."""
    rng = np.random.default_rng(n)
    xy = rng.random((n, 2))
    h = 0.5 * spacings / np.sqrt(n) * (0.7 + 0.3 * rng.random(n))
    rp, col = _search(xy, h, periodic)
    q = np.sort(rng.choice(n, 3000, replace=False))
    orp, ocol = oracle.neighbours_large(xy, h, periodic, queries=q)
    assert np.array_equal(rp[q + 1] - rp[q], np.diff(orp))
    assert np.array_equal(np.concatenate([col[rp[i]:rp[i + 1]] for i in q]), ocol)


def test_row_offsets_of_many_blocks():
    """2898^2 lattice nodes (more than 4,096 blocks of the prefix sum), 2 h = 1.2 spacings: the four nearest nodes,
    fewer at the edges, known without a search."""
    m = 2898
    s = 1.0 / m
    at = np.arange(m * m)
    i, j = at % m, at // m
    xy = np.stack([(i + 0.5) * s, (j + 0.5) * s], 1)
    rp, col = _search(xy, np.full(m * m, 0.6 * s), False)
    near = np.stack([np.where(j > 0, at - m, -1), np.where(i > 0, at - 1, -1), np.where(i < m - 1, at + 1, -1),
                     np.where(j < m - 1, at + m, -1)], 1)
    live = near >= 0
    assert np.array_equal(rp, np.concatenate([[0], np.cumsum(live.sum(1))]))
    assert np.array_equal(col, near[live])
