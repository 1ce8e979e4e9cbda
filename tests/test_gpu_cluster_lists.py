"""Cluster lists where the search takes more than one batch of 128 columns or
of 128 candidate clusters, where most columns in reach are empty (two droplets
apart, a thin row of molecules) and where the ring of queued clusters ends in
a short step, against the FP64 oracle.

Tolerance as for every FP32 pair sum: ||dg_i|| <= 1e-5 of the sum of the
magnitudes of the terms of atom i.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle.forcefield import Params
from oracle.integrate import OracleMD, Topology
from paper_2002_07109_gb300.water import concat_systems, water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


def _ball(n):
    return water_droplet_molecules(n, seed=4)


def _two(n):
    return concat_systems([_ball(n), _ball(n)], spacing=30.0)[0]


def _row(n):
    s = _ball(n)
    s.q = s.q.reshape(-1, 3, 3)
    s.q = (s.q - s.q[:, :1] + 3.1 * np.arange(n)[:, None, None] * np.array([1.0, 0.0, 0.0])).reshape(-1, 3)
    return s


@pytest.mark.parametrize("build, n, r_cut", [(_ball, 300, 9.0), (_ball, 1200, 24.0), (_ball, 1200, 40.0),
                                             (_two, 400, 20.0), (_row, 200, 30.0)])
def test_lists_of_wide_cutoffs(build, n, r_cut):
    s = build(n)
    ctx = bounce.from_system(s, seed=3, r_on=4.0, r_off=5.0, r_cut=r_cut, skin=1.0, max_neighbors=4096)
    ctx.set_state(s.q, s.v)
    p = Params(r_on=4.0, r_off=5.0, r_cut=r_cut, lj_sigma=s.lj_sigma, lj_eps=s.lj_eps)
    topo = Topology(s.type, s.mass, s.charge, s.molecule, s.bonds, s.bond_k_r0, s.angles, s.angle_k_t0)
    md = OracleMD(s.q, s.v, topo, p, seed=3, skin=1.0)
    md.ensure_rows()
    for part, code, ref in (("full", bounce.GRAD_FULL, md.grad_full()), ("short", bounce.GRAD_SHORT, md.grad_short())):
        d = np.linalg.norm(ctx.gradient(code) - ref, axis=1)
        bad = d / np.maximum(md.grad_scale(part), 1e-30)
        assert bad.max() < 1e-5, (part, bad.max(), int(bad.argmax()))
    ctx.close()
