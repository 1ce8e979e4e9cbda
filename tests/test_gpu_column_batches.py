"""Cluster lists of periodic boxes whose search takes its columns in batches
of 128 with no empty one among them (every column of the box, and rows of
columns that wrap), and of a box with just fewer columns in all, against the
FP64 oracle.  Molecules far apart, about eight to a column of 12 A, make wide
searches cheap.

Tolerance as for every FP32 pair sum: ||dg_i|| <= 1e-5 of the sum of the
magnitudes of the terms of atom i.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle.forcefield import (Params, bonded_gradient_magnitudes, bonded_gradients, pair_gradient_magnitudes,
                               pair_gradients)
from oracle.integrate import OracleMD, Topology
from oracle.neighbors import rows, to_pairs
from paper_2002_07109_gb300.water import water_box

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


def spread_box(side):
    """side^3 molecules at the sites of a 12.05 x 12.05 x 18 A lattice, each within 2.5 A of its site on every axis."""
    s = water_box(side, seed=5)
    step = np.array([12.05, 12.05, 18.0])
    g = np.arange(side) + 0.5
    sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) * step
    q = s.q.reshape(-1, 3, 3)
    jitter = np.random.default_rng(6).uniform(-2.5, 2.5, sites.shape)
    s.q = (q - q[:, :1] + (sites + jitter)[:, None]).reshape(-1, 3)
    s.box = side * step
    return s


def _topology(s):
    return Topology(s.type, s.mass, s.charge, s.molecule, s.bonds, s.bond_k_r0, s.angles, s.angle_k_t0)


# 121 columns, 144 (all in reach of each), and 12 or 13 of 14 a row in reach
@pytest.mark.parametrize("side, r_cut", [(11, 62.0), (12, 62.0), (14, 64.0)])
def test_full_batches_of_columns(side, r_cut):
    """The full sums (no pair of these molecules lies within the switch: F_0 has no pair term here)."""
    s = spread_box(side)
    ctx = bounce.from_system(s, seed=3, r_on=4.0, r_off=5.0, r_cut=r_cut, skin=1.0, pair_skin=2.0, max_neighbors=4096)
    ctx.set_state(s.q, s.v)
    p = Params(r_on=4.0, r_off=5.0, r_cut=r_cut, box=s.box, lj_sigma=s.lj_sigma, lj_eps=s.lj_eps)
    md = OracleMD(s.q, s.v, _topology(s), p, seed=3, skin=1.0)
    md.ensure_rows()
    d = np.linalg.norm(ctx.gradient(bounce.GRAD_FULL) - md.grad_full(), axis=1)
    bad = d / np.maximum(md.grad_scale("full"), 1e-30)
    assert bad.max() < 1e-5, (bad.max(), int(bad.argmax()))
    ctx.close()


def test_full_batches_in_water():
    """Water at its density (144 columns, all in reach): full and short sums of the atoms of the first columns, whose
    search meets no empty column, and of atoms drawn anywhere."""
    s = water_box(17, seed=0)
    r_cut = 22.0
    ctx = bounce.from_system(s, seed=3, r_on=4.0, r_off=5.0, r_cut=r_cut, skin=1.0, pair_skin=3.0, max_neighbors=6144)
    ctx.set_state(s.q, s.v)
    p = Params(r_on=4.0, r_off=5.0, r_cut=r_cut, box=s.box, lj_sigma=s.lj_sigma, lj_eps=s.lj_eps)
    first = np.nonzero((s.q[:, :2] % s.box[:2] < 8.0).all(1))[0]
    at = np.union1d(first, np.random.default_rng(1).choice(s.n_atoms, 150, replace=False))
    ii, jj = to_pairs(rows(s.q, s.molecule, r_cut, s.box, at), at)
    bonded = s.bonds, s.bond_k_r0, s.angles, s.angle_k_t0, s.box
    for part, code in (("full", bounce.GRAD_FULL), ("short", bounce.GRAD_SHORT)):
        ref = pair_gradients(s.q, s.charge, s.type, ii, jj, p, part) + bonded_gradients(s.q, *bonded)
        scale = pair_gradient_magnitudes(s.q, s.charge, s.type, ii, jj, p, part) + bonded_gradient_magnitudes(s.q, *bonded)
        bad = np.linalg.norm(ctx.gradient(code) - ref, axis=1)[at] / scale[at]
        assert bad.max() < 1e-5, (part, bad.max(), int(at[bad.argmax()]))
    ctx.close()
