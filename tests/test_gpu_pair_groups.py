"""Edges of the packed pair kernels (two pairs per instruction, groups of
eight i atoms): systems smaller than one group, list and group remainders,
atoms of a group that do not exist, boxes so small that most entries take the
minimum image per pair, the step switch, against the FP64 oracle.

Tolerance as for every FP32 pair sum: ||dg_i|| <= 1e-5 of the sum of the
magnitudes of the terms of atom i.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle.forcefield import Params
from oracle.integrate import OracleMD, Topology
from paper_2002_07109_gb300.water import water_box, water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")

TOL = 1e-5
DROP = dict(r_on=4.0, r_off=5.0, skin=1.0)


@pytest.mark.parametrize("cfg", [dict(DROP, r_cut=8.0), dict(DROP, r_cut=8.0, jump_coulomb=False),
                                 dict(DROP, r_off=4.0, r_cut=8.0), dict(DROP, r_cut=math.inf, jump_coulomb=False)],
                         ids=["cut", "cut_vdw", "cut_step", "all"])
@pytest.mark.parametrize("n_mol", [1, 2, 3, 11, 43, 86])
def test_small_droplets(n_mol, cfg):
    _check(water_droplet_molecules(n_mol, seed=n_mol), cfg)


@pytest.mark.parametrize("side, r_cut", [(6, 9.0), (7, 9.0), (8, 8.0), (9, 9.0)])
@pytest.mark.parametrize("vdw", [False, True], ids=["coulomb_jumps", "vdw_jumps"])
def test_small_boxes(side, r_cut, vdw):
    _check(water_box(side, seed=side), dict(r_on=6.0, r_off=7.0, r_cut=r_cut, skin=0.2, ewald_beta=0.35,
                                            max_neighbors=1024, jump_coulomb=not vdw))


def test_paired_tiles_equal_single_tiles():
    """A batch large enough that two i-tiles share an item gives, bit for bit,
    the pair sums of each droplet alone (one tile an item): tile and block
    remainders of 1 to 31 atoms, replicas of one tile, of one block, of an odd
    number of blocks."""
    from paper_2002_07109_gb300.water import concat_systems
    sizes = [1, 10, 11, 21, 22, 43, 64, 85, 107] * 20
    cat, off = concat_systems([water_droplet_molecules(m, seed=m) for m in sizes], spacing=0.0)
    cfg = dict(DROP, jump_coulomb=False, max_neighbors=400)
    ctx = bounce.from_system(cat, seed=1, **cfg)
    ctx.set_replicas(off, np.arange(len(sizes), dtype=np.uint64))
    ctx.set_state(cat.q, cat.v)
    both = [ctx.gradient(code) for code in (bounce.GRAD_FULL, bounce.GRAD_SHORT)]
    ctx.close()
    for r, m in enumerate(sizes[:9]):
        s = water_droplet_molecules(m, seed=m)
        one = bounce.from_system(s, seed=1, **cfg)
        one.set_state(s.q, s.v)
        for g, code in zip(both, (bounce.GRAD_FULL, bounce.GRAD_SHORT)):
            ref = one.gradient(code)
            for k in range(r, len(sizes), 9):
                assert np.array_equal(g[off[k]:off[k + 1]], ref), (m, k, code)
        one.close()


def _check(s, cfg):
    q = s.q + np.random.default_rng(7).normal(scale=0.05, size=s.q.shape) + 1.3   # some atoms outside the box
    ctx = bounce.from_system(s, seed=3, **cfg)
    ctx.set_state(q, s.v)
    p = Params(r_on=cfg["r_on"], r_off=cfg["r_off"], r_cut=cfg["r_cut"], ewald_beta=cfg.get("ewald_beta", 0.0),
               box=s.box, lj_sigma=s.lj_sigma, lj_eps=s.lj_eps, coulomb_jumps=cfg.get("jump_coulomb", True))
    topo = Topology(s.type, s.mass, s.charge, s.molecule, s.bonds, s.bond_k_r0, s.angles, s.angle_k_t0)
    md = OracleMD(q, s.v, topo, p, seed=3, skin=cfg["skin"])
    md.ensure_rows()
    for part, code, ref in (("full", bounce.GRAD_FULL, md.grad_full()), ("short", bounce.GRAD_SHORT, md.grad_short())):
        d = np.linalg.norm(ctx.gradient(code) - ref, axis=1)
        bad = d / np.maximum(md.grad_scale(part), 1e-30)
        assert bad.max() < TOL, (part, bad.max(), int(bad.argmax()))
    ctx.close()
