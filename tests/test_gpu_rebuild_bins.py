"""The binning of the atoms (one cluster of eight CTAs for the cells, one for
the columns) and the lists built in the same launch as their prune, at atom
counts around the threads' passes: rebuilds inside runs give the lists that a
state set at the same positions gets, in bits of the fixed-point pair sums.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2002_07109_gb300.water import water_box, water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


@pytest.mark.parametrize("n_mol, integ", [(1, "BOUNCE"), (342, "BOUNCE"), (2730, "BAOAB"), (2731, "BOUNCE"),
                                          (10923, "BOUNCE")])
def test_droplet_rebuilt_in_a_run(n_mol, integ):
    """Atoms of a droplet keep their coordinates, so that the pair sums of the two contexts are the same terms."""
    s = water_droplet_molecules(n_mol, seed=3)
    cfg = dict(seed=2, jump_coulomb=False, r_on=4.0, r_off=5.0, r_cut=8.0, skin=0.3, pair_skin=0.3, max_neighbors=1024)
    a, b = bounce.from_system(s, **cfg), bounce.from_system(s, **cfg)
    a.set_state(s.q, s.v, step=0)
    a.run(30, getattr(bounce, integ))
    if n_mol > 1 and integ == "BOUNCE":
        assert a.energies()["rebuilds"] > 2
    b.set_state(*a.get_state(), step=30)
    for part in (bounce.GRAD_FULL, bounce.GRAD_SHORT):
        assert np.abs(a.gradient(part) - b.gradient(part)).max() <= 1e-5 * np.abs(b.gradient(part)).max()
    assert all(np.array_equal(x, y) for x, y in zip(a.rows(), b.rows()))
    a.close()
    b.close()


def test_box_runs_repeat_with_either_skin():
    """A box whose clusters are rebuilt at nearly every prune, and one where prunes alone occur: the pairs inside the
    cutoff are the same."""
    s = water_box(12, seed=3)
    out = []
    for pair_skin in (0.25, 2.0):
        ctx = bounce.from_system(s, seed=2, jump_coulomb=False, r_on=6.0, r_off=7.0, r_cut=8.0, skin=1.0,
                                 pair_skin=pair_skin, ewald_beta=0.35, max_neighbors=1024)
        ctx.set_state(s.q, s.v, step=0)
        ctx.run(20, bounce.BAOAB)
        out.append(ctx.get_state())
        ctx.close()
    assert np.abs(out[0][0] - out[1][0]).max() < 1e-4
