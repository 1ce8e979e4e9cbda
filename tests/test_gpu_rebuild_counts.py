"""Lists that were rebuilt inside a run hold the same pairs as the lists of a
state set afresh at the same positions: the pairs that the sums count inside
the cutoff are equal, to the last one.  That rebuilds were due shows in the
displacement from the first positions.  (Droplets: the coordinates, and so the
exact cutoff test of every pair, are the same in both contexts.)
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2002_07109_gb300.water import water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")

SKIN = 0.3


def pairs_counted(ctx):
    out = []
    for part, key in ((bounce.GRAD_FULL, "full_pairs"), (bounce.GRAD_SHORT, "short_pairs")):
        ctx.reset_counters()
        ctx.gradient(part)
        out.append(ctx.energies()[key])
    return out


@pytest.mark.parametrize("n_mol, integ", [(342, "BOUNCE"), (2730, "BAOAB"), (2731, "BOUNCE"), (10923, "BAOAB")])
def test_pairs_of_rebuilt_lists(n_mol, integ):
    s = water_droplet_molecules(n_mol, seed=3)
    cfg = dict(seed=2, jump_coulomb=False, r_on=4.0, r_off=5.0, r_cut=8.0, skin=SKIN, pair_skin=SKIN, max_neighbors=1024)
    a, b = bounce.from_system(s, **cfg), bounce.from_system(s, **cfg)
    a.set_state(s.q, s.v, step=0)
    a.run(30, getattr(bounce, integ))
    q, v = a.get_state()
    assert (((q - s.q) ** 2).sum(1) > SKIN ** 2).any()      # twice the half skin that calls for a rebuild
    b.set_state(q, v, step=30)
    counts = pairs_counted(a)
    assert counts == pairs_counted(b) and min(counts) > 0
    a.close()
    b.close()
