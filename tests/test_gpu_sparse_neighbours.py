"""Neighbour search where bins hold an atom or two and runs of them share a work item, and where lists are long."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle.neighbours import neighbour_list  # noqa: E402
from synth import System  # noqa: E402


@pytest.fixture(scope="module")
def rg():
    import paper_2101_08814_gb300 as rg

    return rg


def _lists(rg, s, r_cut):
    calc = rg.SoapCalculator(r_cut, 0.5, 2, 1, [6], spline_intervals=64)
    pl = calc.neighbours(rg.DeviceSystem.from_numpy(s))
    return [getattr(pl, k).cpu().numpy() for k in ("offsets", "nbr_j", "shifts", "rij")]


def _system(pos, cells, pbc, sizes):
    n = len(sizes)
    return System(pos, np.full(len(pos), 6, np.int32), np.asarray(cells, float), np.tile(np.asarray([pbc], np.int32), (n, 1)),
                  np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), {})


# Runs along the third axis: sparse all over, sparse with one crowded corner (its bins are parts of a run that splits into several
# items), a short third axis (runs of one bin, several images), a triclinic cell, an open third axis, vacuum around a cluster, 70
# structures of a few atoms each. Equal to the brute-force list.
@pytest.mark.parametrize("case", ["sparse", "corner", "flat", "triclinic", "open", "cluster", "molecules"])
def test_runs_of_sparse_bins(rg, case):
    rng = np.random.default_rng(97)
    cell, pbc, n, r_cut = np.eye(3) * 24.0, (1, 1, 1), 300, 3.0
    if case == "flat":
        cell, n = np.diag([30.0, 30.0, 4.0]), 150
    if case == "triclinic":
        cell = np.array([[22.0, 0.0, 0.0], [6.0, 21.0, 0.0], [-5.0, 4.0, 23.0]])
    if case == "open":
        pbc = (1, 1, 0)
    pos = rng.random((n, 3)) @ cell
    if case == "corner":
        pos[:60] = rng.random((60, 3)) * 2.9
    if case == "cluster":
        cell, pos = np.eye(3) * 60.0, 25.0 + rng.random((n, 3)) * 9.0
    cells, sizes = cell[None], [n]
    if case == "molecules":
        sizes = rng.integers(0, 9, 70)
        pos = rng.random((int(sizes.sum()), 3)) * 5.0
        cells = np.tile(np.diag([9.0, 10.0, 14.0])[None], (70, 1, 1))
    s = _system(pos, cells, pbc, sizes)
    off, j, sh, rij = _lists(rg, s, r_cut)
    ref = neighbour_list(s, r_cut)
    assert np.array_equal(off, ref["offsets"]) and np.array_equal(j, ref["nbr_j"]) and np.array_equal(sh, ref["shifts"])
    assert np.allclose(rij[:, :3], ref["rij"], rtol=0, atol=2e-6)


# One structure with more bins than one pass of the scan takes (8 192): against a periodic k-d tree
def test_many_bins(rg):
    from scipy.spatial import cKDTree

    rng = np.random.default_rng(101)
    L, n, r_cut = 90.0, 9000, 3.0
    pos = rng.random((n, 3)) * L
    off, j, sh, _ = _lists(rg, _system(pos, np.eye(3)[None] * L, (1, 1, 1), [n]), r_cut)
    found = cKDTree(pos, boxsize=L).query_ball_point(pos, r_cut)
    want = [sorted(k for k in f if k != i) for i, f in enumerate(found)]
    assert np.array_equal(np.diff(off), [len(w) for w in want])
    assert np.array_equal(j, np.concatenate(want))
    d = pos[j] - pos[np.repeat(np.arange(n), np.diff(off))] + sh * L
    assert np.all((d ** 2).sum(1) < r_cut ** 2)


# Lists of 129 to 256 pairs per centre are sorted in shared memory as in the no-allocation search, longer ones in scratch
@pytest.mark.parametrize("n,r_cut,low,high", [(160, 5.2, 129, 256), (240, 6.6, 257, 900)])
def test_long_lists(rg, n, r_cut, low, high):
    rng = np.random.default_rng(103)
    L = 9.5 if n == 160 else 10.0
    s = _system(rng.random((n, 3)) * L * 0.8, np.eye(3)[None] * L, (1, 1, 1), [n])
    off, j, sh, rij = _lists(rg, s, r_cut)
    ref = neighbour_list(s, r_cut)
    assert np.array_equal(off, ref["offsets"]) and np.array_equal(j, ref["nbr_j"]) and np.array_equal(sh, ref["shifts"])
    assert low <= np.diff(off).max() <= high
