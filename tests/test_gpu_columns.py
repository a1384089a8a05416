"""Radial rows of the coefficients-only call: lanes over the table's columns, written to padded slots."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from synth import System, random_cell_atoms  # noqa: E402


# The fused call fills its rows over the padded slots: coefficients alone are the same bits. n_max of every remainder by 4, from
# 1 to 32 (a row of 32 columns of one l), fewer columns than lanes and several turns of them, an odd number of rows, compiled
# shapes and not, one species round and several; DVR, whose basis stays regular at the widest n_max.
@pytest.mark.parametrize("n_max,l_max,S", [(1, 0, 1), (1, 15, 2), (2, 3, 3), (3, 0, 1), (6, 6, 2), (7, 15, 1), (8, 5, 3), (10, 8, 3),
                                           (11, 4, 9), (13, 9, 2), (30, 2, 3), (31, 2, 3), (32, 3, 2)])
def test_coefficients_over_table_columns(n_max, l_max, S):
    import torch

    import paper_2101_08814_gb300 as rg

    calc = rg.SoapCalculator(4.5, 0.5, n_max, l_max, list(range(1, S + 1)), basis="dvr", spline_intervals=64)
    rng = np.random.default_rng(79)
    n = 65
    L = (n / 0.11) ** (1 / 3)
    s = System(np.concatenate([random_cell_atoms(n, np.eye(3) * L, 0.9, rng), [[0.0, 0.0, 60.0]]]),
               rng.integers(1, S + 1, n + 1).astype(np.int32), np.diag([L, L, 200.0])[None], np.array([[1, 1, 0]], np.int32),
               np.array([0, n + 1], np.int32), {})
    ds = rg.DeviceSystem.from_numpy(s)
    pairs = calc.neighbours(ds)
    counts = np.diff(pairs.offsets.cpu().numpy())
    assert counts.max() > 32 and np.any(counts % 2 == 1) and counts[-1] == 0
    ref, _ = calc.soap(ds, pairs)
    c = calc.spherical_expansion(ds, pairs)
    assert bool(torch.isfinite(ref).all()) and torch.equal(c, ref)
