"""The pair lists behind H, gamma and the forces at the sizes where they can go wrong: atom
counts around the rows of a block (one row below 128 atoms, two from 128, sixteen from 1024)
and the 256 columns of a block, in boxes above twice the interaction range (only the nearest
image) and below it (every image).

All FP64 on both sides: the tolerances cover the rounding of exp and sqrt and the order of
sums, as for the same comparisons on the other systems."""

import numpy as np
import pytest
import torch

from workloads import ModelParams, water_system
from oracle import observables, tb
from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import DeviceSystem

pytestmark = pytest.mark.gpu
P = ModelParams()
TP = tbmd.tb_params.from_model(P)


@pytest.mark.parametrize("density", [0.02, 1.0])
@pytest.mark.parametrize("natoms", [3, 127, 128, 255, 257, 1025])
def test_H_gamma_and_forces_at_the_edges_of_the_pair_lists(ctx, natoms, density):
    s = water_system(natoms, density=density, seed=natoms)
    N = s.natoms
    rng = np.random.default_rng(natoms)
    n_aux = rng.normal(0, 0.2, N)
    q = rng.normal(0, 0.2, N)
    ds = DeviceSystem(s.R, s.types, s.box)
    n = ds.norb
    H = torch.empty(n, n, dtype=torch.float64, device="cuda")
    G = torch.empty(N, N, dtype=torch.float64, device="cuda")
    F = torch.empty(N, 3, dtype=torch.float64, device="cuda")
    E = torch.empty(4, dtype=torch.float64, device="cuda")
    A = rng.normal(0, 0.1, (n, n))
    D = 0.5 * (A + A.T)
    nt = torch.as_tensor(n_aux, device="cuda")
    tbmd.tb_build_H(ctx, TP, ds.sys, ds.R, nt, H, G)
    tbmd.tb_forces(ctx, TP, ds.sys, ds.R, torch.as_tensor(D, device="cuda"), torch.as_tensor(q, device="cuda"), nt, G,
                   F, E)
    torch.cuda.synchronize()
    Go = tb.build_gamma(s.R, s.box, P)
    Ho = tb.build_H(tb.build_h(s.R, s.types, s.box, P), Go, s.types, n_aux)
    assert np.abs(G.cpu().numpy() - Go).max() < 1e-11
    assert np.abs(H.cpu().numpy() - Ho).max() < 1e-11
    Fo = observables.forces(s.R, s.types, s.box, P, D, q, n_aux)
    assert np.abs(F.cpu().numpy() - Fo).max() < 1e-9 * max(1.0, np.abs(Fo).max())
