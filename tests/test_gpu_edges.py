"""Launch forms at the sizes where they change: the Newton-Schulz iteration of the
non-orthogonal step (one launch up to n = 512, a sequence above), and the closing kick and
kinetic energy of an MD step (one block up to 512 atoms, a cluster of eight above)."""

import numpy as np
import pytest
import torch

from workloads import XLParams, gapped_params, gapped_vapour, random_gapped_matrix, thermal_velocities
from oracle import nonorth, observables
from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import DeviceSystem, MDState, NonorthSolver, nonorth_report_to_dict, sp2_opts, \
    xl_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 33, 129, 512, 513])
def test_dm_nonorth_sizes(ctx, n):
    H, _ = random_gapped_matrix(n, n // 2, gap=2.0, width=20.0, seed=n)
    rng = np.random.default_rng(n)
    B = rng.normal(size=(n, n))
    B = 0.5 * (B + B.T)
    S = np.eye(n) + 0.3 * B / np.abs(np.linalg.eigvalsh(B)).max()  # eigenvalues within 0.7 .. 1.3
    ref = nonorth.density_matrix(H, S, n // 2)
    rho = torch.empty(n, n, dtype=torch.float64, device="cuda")
    W = torch.empty_like(rho)
    sol = NonorthSolver(ctx, n, 0.0, sp2=sp2_opts("fp64", tol=1e-11))
    sol(torch.as_tensor(H, device="cuda"), torch.as_tensor(S, device="cuda"), float(n // 2), rho, W)
    torch.cuda.synchronize()
    assert nonorth_report_to_dict(sol.report)["status"] == tbmd.TB_OK
    # the bounds of the same comparison on molecular systems (W carries |H|)
    assert np.linalg.norm(rho.cpu().numpy() - ref.rho) / np.sqrt(n) < 1e-9
    assert np.linalg.norm(W.cpu().numpy() - ref.W) / np.sqrt(n) < 3e-8


@pytest.mark.parametrize("molecules", [1, 170, 171, 172])
def test_kinetic_energy_of_a_step(ctx, molecules):
    p = gapped_params()
    s = gapped_vapour(molecules, seed=1)  # 3, 510, 513 and 516 atoms
    M = s.masses(p)
    ds = DeviceSystem(s.R, s.types, s.box)
    opts = sp2_opts("tf32x3", max_iter=100, refine=2)
    xl = XLParams()
    st = MDState(ds, thermal_velocities(M, 300.0, seed=2), M, s.n_occ(p), xl.K, opts)
    xp = xl_params(xl.dt, xl.kappa, xl.alpha, xl.c)
    tp = tbmd.tb_params.from_model(p)
    tbmd.xlbomd_init(ctx, tp, st.st, xp, opts, 1e-6, 100)
    tbmd.xlbomd_step(ctx, tp, st.st, xp, opts)
    torch.cuda.synchronize()
    e = st.energies.cpu().numpy()
    # FP64 sums of at most 516 positive terms on both sides
    assert e[5] == pytest.approx(observables.kinetic_energy(st.v.cpu().numpy(), M), rel=1e-12)
    assert e[0] == pytest.approx(e[1] + e[5], rel=1e-12)
