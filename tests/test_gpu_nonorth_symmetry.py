"""dm_nonorth's rho and W are exactly symmetric: sizes within one tile, at its edges, with ragged
last tiles, and on both sides of the launched forms' larger tiles (n = 512)."""

import numpy as np
import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import NonorthSolver, fermi_report_to_dict, nonorth_report_to_dict, sp2_opts
from workloads import random_gapped_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kT", [0.0, 0.3])
@pytest.mark.parametrize("n", [2, 15, 16, 17, 129, 384, 512, 513, 600])
def test_rho_and_W_are_symmetric(ctx, n, kT):
    H, _ = random_gapped_matrix(n, n // 2, gap=2.0, width=20.0, seed=n)
    rng = np.random.default_rng(n)
    B = rng.normal(size=(n, n))
    B = 0.5 * (B + B.T)
    S = np.eye(n) + 0.3 * B / np.abs(np.linalg.eigvalsh(B)).max()  # eigenvalues within 0.7 .. 1.3
    S = 0.5 * (S + S.T)
    rho = torch.full((n, n), float("nan"), dtype=torch.float64, device="cuda")
    W = torch.full_like(rho, float("nan"))
    s = NonorthSolver(ctx, n, kT, sp2=sp2_opts("fp64", tol=1e-11))
    s(torch.as_tensor(H, device="cuda"), torch.as_tensor(S, device="cuda"), float(n // 2), rho, W)
    torch.cuda.synchronize()
    assert nonorth_report_to_dict(s.report)["status"] == tbmd.TB_OK
    if kT > 0.0:
        assert fermi_report_to_dict(s.fermi_report)["status"] == tbmd.TB_OK
    assert torch.equal(rho, rho.T.contiguous())
    assert torch.equal(W, W.T.contiguous())
