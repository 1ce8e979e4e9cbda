"""Candidate rows where the row builder's branches change: boxes barely wider
than twice r_list (where the FP32 image can decide a member) and wider ones,
molecules in an order unrelated to their places (members outside the bitmap's
window take further passes), bitmaps of one word up to several passes of 128
words.  Rows are sets of integers: equal to the FP64 oracle's, no tolerance.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle.integrate import typed_rows
from oracle.neighbors import rows as oracle_rows
from paper_2002_07109_gb300.water import water_box, water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


def _check(s, q, r_list, typed, box, sample):
    ctx = bounce.from_system(s, seed=2, pair_bounds=typed, r_on=2.0, r_off=3.0, r_cut=r_list - 0.5, skin=0.5)
    ctx.set_state(q, s.v, step=0)
    got = ctx.rows()
    ctx.close()
    ref = oracle_rows(q, s.molecule, r_list, box, atoms=sample)
    if typed:
        ref, _ = typed_rows(ref, s.type, 2)
    for i, r in zip(sample, ref):
        assert np.array_equal(got[i], r), i


@pytest.mark.parametrize("typed", [False, True])
@pytest.mark.parametrize("n_side, half", [(4, 0.49999), (6, 0.49999), (6, 0.4985), (9, 0.49999), (12, 0.3)])
def test_rows_of_boxes(n_side, half, typed):
    s = water_box(n_side, seed=5)
    q = s.q + np.array([1.3, -40.0, 77.0])
    n = len(q)
    _check(s, q, half * s.box[0], typed, s.box, np.unique(np.linspace(0, n - 1, 400).astype(int)))


@pytest.mark.parametrize("n_mol, typed", [(7, True), (43, True), (342, False), (1366, True), (4500, False), (9000, True)])
def test_rows_in_any_order(n_mol, typed):
    s = water_droplet_molecules(n_mol, seed=3)
    q = s.q.reshape(-1, 3, 3)[np.random.default_rng(1).permutation(n_mol)].reshape(-1, 3)
    _check(s, q, 8.0, typed, None, np.unique(np.linspace(0, len(q) - 1, 300).astype(int)))
