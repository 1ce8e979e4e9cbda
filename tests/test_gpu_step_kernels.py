"""The step kernels where their launch shape and their conversions change:
atom counts on both sides of each CTA size of the cooperative kernel (which
then has 2, 4, 8, 16 or 32 atoms to a CTA) against the thread-per-atom kernel,
whose result does not depend on it, and the split FP32 positions that the step
kernels leave (integer conversions) against those of a state set from outside
(the conversion instructions).  Both are comparisons of bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2002_07109_gb300.water import water_box, water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


@pytest.mark.parametrize("n_mol", [1, 304, 305, 608, 609, 1216, 1217, 2432, 2433])
def test_atoms_of_a_cooperative_cta(n_mol):
    s = water_droplet_molecules(n_mol, seed=4)
    out = []
    for sk in (1, 2):
        ctx = bounce.from_system(s, seed=5, r_on=3.0, r_off=4.0, jump_coulomb=False, max_neighbors=3 * n_mol, step_kernel=sk)
        ctx.set_state(s.q, s.v, step=0)
        ctx.run(3, bounce.BOUNCE)
        e = ctx.energies()
        out.append((*ctx.get_state(), e["proposals"], e["accepts"], e["near_ties"]))
        ctx.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("sk", [1, 2])
@pytest.mark.parametrize("scale", [0.0, 1e-30, 1e-12, 1.0, -3.0e5])
def test_split_positions_of_a_step(sk, scale):
    """Offsets: a molecule at the origin itself (zeros), at subnormal and at tiny distances of it, and far off."""
    s = water_droplet_molecules(40, seed=6)
    q = s.q - s.q[0] + scale * np.array([1.0, -1.0, 0.5])
    v = np.zeros_like(s.v)
    v[60:] = s.v[60:]
    cfg = dict(seed=5, jump_coulomb=False, r_on=4.0, r_off=5.0, dt=1e-3, gamma=0.0, step_kernel=sk)
    a, b = bounce.from_system(s, **cfg), bounce.from_system(s, **cfg)
    a.set_state(q, v, step=0)
    a.run(2, bounce.BAOAB)
    b.set_state(*a.get_state(), step=2)
    for part in (bounce.GRAD_FULL, bounce.GRAD_SHORT, bounce.GRAD_LONG):
        assert np.array_equal(a.gradient(part), b.gradient(part))
    a.close()
    b.close()


@pytest.mark.parametrize("sk", [1, 2])
def test_split_positions_in_a_box(sk):
    """Atoms on both sides of the faces and several edges away from the box."""
    s = water_box(6, seed=6)
    L = s.box[0]
    rng = np.random.default_rng(2)
    mol = np.arange(len(s.q)) // 3
    q = s.q + (rng.integers(-3, 4, (mol.max() + 1, 3)) * L)[mol] + np.array([0.5 * L, -L / 3, 1e-9])
    cfg = dict(seed=5, r_on=4.0, r_off=5.0, r_cut=0.45 * L, skin=0.5, ewald_beta=0.35, step_kernel=sk)
    a, b = bounce.from_system(s, **cfg), bounce.from_system(s, **cfg)
    a.set_state(q, s.v, step=0)
    a.run(3, bounce.BAOAB)
    b.set_state(*a.get_state(), step=3)
    assert np.array_equal(a.energies()["bond"], b.energies()["bond"])
    assert all(np.array_equal(x, y) for x, y in zip(a.rows(), b.rows()))
    a.close()
    b.close()
