"""The SPME passes by the kind of the grid's axes, against the FP64 oracle:
planes of lines of 32 M points, planes of other products of 2, 3, 4 and 5
(also narrower than the padding of the gather's rows), axes of mixed kinds and
axes with another prime factor; every spline order (the spread shares an atom
among as many lanes, with a last CTA that is not full).

Tolerance as for every FP32 sum: the error of atom i against 1e-5 of the
magnitudes of its two parts (reciprocal and same-molecule); energies 1e-6 of
the sum of the magnitudes of their parts.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import ewald
from paper_2002_07109_gb300.water import water_box

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")

GRIDS = [(32, 32, 32), (64, 64, 64), (96, 32, 32), (24, 24, 24), (45, 36, 40), (8, 9, 10), (64, 48, 64), (48, 64, 64),
         (34, 32, 32), (33, 33, 33)]


@pytest.mark.parametrize("grid, order", [(g, 5) for g in GRIDS] + [((32, 32, 32), n) for n in (3, 4, 6, 7, 8)] +
                         [((27, 27, 27), n) for n in (3, 8)])
def test_recip_by_grid_kind(grid, order):
    s = water_box(6, seed=2)
    q = s.q + 2.9
    ctx = bounce.from_system(s, r_on=4.0, r_off=5.0, r_cut=9.0, ewald_beta=0.35, skin=0.2, max_neighbors=1024,
                             pme_grid=grid, pme_order=order)
    ctx.set_state(q, s.v)
    g = ctx.gradient(bounce.GRAD_RECIP)
    assert np.array_equal(g, ctx.gradient(bounce.GRAD_RECIP))       # the grid is left clear
    e = ctx.energies()["recip"]
    assert np.array_equal(g, ctx.gradient(bounce.GRAD_RECIP))       # also by the energy evaluation
    ctx.close()
    er, gr = ewald.spme_recip(q, s.charge, s.box, 0.35, grid, order)
    ex, gx = ewald.exclusion(q, s.charge, ewald.molecule_pairs(s.molecule), 0.35, s.box)
    es = ewald.self_energy(s.charge, 0.35)
    assert abs(e - (er + ex + es)) <= 1e-6 * (abs(er) + abs(ex) + abs(es))
    scale = np.linalg.norm(gr, axis=1) + np.linalg.norm(gx, axis=1)
    d = np.linalg.norm(g - (gr + gx), axis=1)
    assert (d <= 1e-5 * scale).all(), (d / scale).max()
