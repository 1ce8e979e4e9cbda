"""SPME grids whose third axis is shorter than the eight points of padding
before the gather's rows, so that the padding holds several periods of a row:
planes of stages, axis by axis with another prime factor, and axes of mixed
kinds, against the FP64 oracle.

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


@pytest.mark.parametrize("grid, order", [((8, 9, 5), 5), ((9, 8, 6), 5), ((10, 6, 7), 5), ((32, 32, 5), 5), ((8, 6, 3), 3)])
def test_recip_with_a_short_third_axis(grid, order):
    s = water_box(6, seed=2)
    q = s.q + 1.7
    ctx = bounce.from_system(s, r_on=4.0, r_off=5.0, r_cut=9.0, ewald_beta=0.35, skin=0.2, max_neighbors=1024,
                             pme_grid=grid, pme_order=order)
    ctx.set_state(q, s.v)
    g, e = ctx.gradient(bounce.GRAD_RECIP), ctx.energies()["recip"]
    ctx.close()
    er, gr = ewald.spme_recip(q, s.charge, s.box, 0.35, grid, order)
    ex, gx = ewald.exclusion(q, s.charge, ewald.molecule_pairs(s.molecule), 0.35, s.box)
    es = ewald.self_energy(s.charge, 0.35)
    assert abs(e - (er + ex + es)) <= 1e-6 * (abs(er) + abs(ex) + abs(es))
    scale = np.linalg.norm(gr, axis=1) + np.linalg.norm(gx, axis=1)
    d = np.linalg.norm(g - (gr + gx), axis=1)
    assert (d <= 1e-5 * scale).all(), (d / scale).max()
