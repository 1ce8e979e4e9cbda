"""The all-pairs tiles under periodic boundaries (no cutoff: every pair under
its minimum image), with one and with two i-tiles to an item, against the FP64
oracle; atoms of a negative molecule take no part in the tiles' sums.  In boxes
of these edges the minimum image of a coordinate far outside the box, where
such atoms and the lanes without an atom are placed, is near 0.

Positions lie on a grid of which half the box is an odd number of half steps,
so that no pair is near a change of its image.  Tolerance as for every FP32
pair sum: ||dg_i|| <= 1e-5 of the sum of the magnitudes of the terms of atom i.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle.forcefield import Params
from oracle.integrate import OracleMD, Topology
from paper_2002_07109_gb300.water import water_box

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


def grid_box(side, edge):
    """side^3 molecules in a cube of the given edge, coordinates on a grid of step edge / 2001."""
    s = water_box(side, seed=9)
    q = s.q.reshape(-1, 3, 3)
    q = q + q[:, :1] * (edge / s.box - 1.0)
    h = edge / 2001
    s.q = np.round(q.reshape(-1, 3) / h) * h
    s.box = np.full(3, edge)
    return s


def check(s, p, ctx, of):
    """Sums of the atoms `of` against those of the system of these atoms alone."""
    n = len(of)
    md = OracleMD(s.q[of], s.v[of], Topology(s.type[of], s.mass[of], s.charge[of], s.molecule[of], s.bonds[:2 * n // 3],
                                             s.bond_k_r0[:2 * n // 3], s.angles[:n // 3], s.angle_k_t0[:n // 3]), p, seed=3)
    md.ensure_rows()
    for part, code, ref in (("full", bounce.GRAD_FULL, md.grad_full()), ("short", bounce.GRAD_SHORT, md.grad_short())):
        bad = np.linalg.norm(ctx.gradient(code)[of] - ref, axis=1) / md.grad_scale(part)
        assert bad.max() < 1e-5, (part, bad.max(), int(bad.argmax()))


# 1,536 atoms: one i-tile to an item; 3,000: two
@pytest.mark.parametrize("side, edge, beta, out", [(8, 32.0, 0.0, None), (10, 32.0, 0.0, None), (10, 32.0, 0.35, None),
                                                   (10, 35.2, 0.0, None), (8, 32.0, 0.0, 5), (10, 32.0, 0.0, 5),
                                                   (10, 35.2, 0.35, 5)])
def test_periodic_tiles(side, edge, beta, out):
    s = grid_box(side, edge)
    of = np.arange(s.n_atoms)
    if out is not None:
        s.molecule[s.molecule == out] = -1
        of = of[s.molecule >= 0]
    ctx = bounce.from_system(s, seed=3, r_on=4.0, r_off=5.0, r_cut=math.inf, ewald_beta=beta, jump_coulomb=False,
                             max_neighbors=4096)
    ctx.set_state(s.q, s.v)
    check(s, Params(r_on=4.0, r_off=5.0, ewald_beta=beta, box=s.box, lj_sigma=s.lj_sigma, lj_eps=s.lj_eps,
                    coulomb_jumps=False), ctx, of)
    ctx.close()
