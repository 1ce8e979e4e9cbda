"""Allocation-free pair energies at the edges of the blocks of 64 atoms: one
block, odd and even numbers of blocks (of the even ones the last distance is
met from one side only), remainders, an LJ table that is not symmetric, against
a direct FP64 sum.  Tolerance as for every FP32 pair energy: 1e-6 of the sum of
the magnitudes of the terms.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2002_07109_gb300.water import water_droplet_molecules

bounce = pytest.importorskip("paper_2002_07109_gb300.bounce")


@pytest.mark.parametrize("n_mol", [1, 21, 22, 42, 43, 64, 85, 107, 171])
def test_blocks(n_mol):
    s = water_droplet_molecules(n_mol, seed=2)
    sig, eps = np.array([[3.1, 1.2], [0.7, 0.4]]), np.array([[0.15, 0.02], [0.05, 0.01]])
    dev = torch.device("cuda", 0)
    out = torch.full((2,), float("nan"), dtype=torch.float64, device=dev)
    r = bounce.pair_energy_noalloc(
        torch.tensor(s.q, device=dev), torch.tensor(s.charge, dtype=torch.float64, device=dev),
        torch.tensor(s.type, dtype=torch.int32, device=dev), torch.tensor(s.molecule, dtype=torch.int32, device=dev),
        sig, eps, float("inf"), 0.0, None, out, torch.cuda.current_stream(dev).cuda_stream)
    assert r == 0
    i, j = np.triu_indices(len(s.q), 1)
    i, j = (x[s.molecule[i] != s.molecule[j]] for x in (i, j))
    d = np.linalg.norm(s.q[i] - s.q[j], axis=1)
    c = 332.063713 * s.charge[i] * s.charge[j] / d
    x = (sig[s.type[i], s.type[j]] / d) ** 6
    rep, att = 4 * eps[s.type[i], s.type[j]] * x * x, 4 * eps[s.type[i], s.type[j]] * x
    got = out.cpu().numpy()
    assert abs(got[0] - c.sum()) <= 1e-6 * np.abs(c).sum() + 1e-9
    assert abs(got[1] - (rep - att).sum()) <= 1e-6 * (rep + att).sum() + 1e-9
