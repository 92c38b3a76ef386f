"""The cell counts' scan where the cells fill thousands of blocks: dilute boxes.

The starts are exact, and the binning's time grows with the cells, not with their square: a box
of eight times the cells may take twelve times as long (eight for work that is linear, and half as
much again for what caches and launches make of it; sums over all blocks before each block, which
are quadratic, made it eighteen times).
"""
import numpy as np
import pytest
import torch

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def handle(N, L, frac=0.5):
    """Cells of edge 1, cell_sub 1: L^3 of them."""
    sy = synth.make_system(N, L=L, seed=9, frac_charged=frac, sigma=0.3)
    return sy, binding.from_system(sy, P=4, alpha=1.0, r_c=1.0, cell_sub=1)


@pytest.mark.parametrize("L", [12.5, 13.0, 60.0, 160.0, 300.0, 330.0])
def test_starts_are_exact(L):
    """One block of cells, two, some hundred, 2,000 (one past a round of the totals' own pass),
    13,000, and 17,000, where that pass runs."""
    N = 20001
    sy, h = handle(N, L)
    with h:
        h.forces(0)
        n, start, ids = h.cells()
    assert tuple(n) == (int(L),) * 3
    c = (sy.s.astype(np.int64) * np.asarray(n, np.int64)) >> 32
    key = c[:, 0] + n[0] * (c[:, 1] + np.int64(n[1]) * c[:, 2])
    count = np.bincount(key, minlength=int(L) ** 3)
    assert np.array_equal(start, np.concatenate([[0], np.cumsum(count)]))
    assert np.array_equal(np.sort(ids), np.arange(N))
    assert np.array_equal(key[ids], np.sort(key))


def test_time_is_linear_in_the_cells():
    def binning(L):
        _, h = handle(2000, L)
        with h:
            h.set_profiling(True)
            ms = []
            for _ in range(4):
                h.forces(0)
                ms.append(h.profile()[0]["bin"])
        return min(ms[1:])
    assert binning(1200.0) < 12.0 * binning(600.0)


def test_batch_of_dilute_boxes():
    """Two boxes whose totals have a pass of their own, stepped as a batch and alone."""
    def two():
        return [handle(n, 330.0)[1] for n in (2000, 3001)]
    alone, together = two(), two()
    for h in alone:
        h.step(2)
    b = binding.Batch(together)
    b.step(2)
    torch.cuda.synchronize()
    for x, y in zip(alone, together):
        assert np.array_equal(x.state()[2], y.state()[2])
        assert np.array_equal(x.cells()[1], y.cells()[1])
    b.close()
    for h in alone + together:
        h.close()
