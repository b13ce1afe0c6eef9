"""The block lists of the block-sparse products at the sizes where they can go wrong: one
super-row, a last band of one row and a padded last row, and two bitmap words.

H couples groups of eight orbitals spread evenly over the matrix, so each super-row has
blocks far from the diagonal and the pattern is closed under products: D is the groups'
own, and the block products of every projection can be counted from H's pattern."""

import numpy as np
import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import DensitySolver, report_to_dict, sp2_opts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", [1, 16, 129, 525])
def test_products_of_a_pattern_far_from_the_diagonal(ctx, groups):
    n = 8 * groups
    rng = np.random.default_rng(groups)
    H, D = np.zeros((n, n)), np.zeros((n, n))
    for g in range(groups):
        Q, _ = np.linalg.qr(rng.normal(size=(8, 8)))
        w = np.concatenate([rng.uniform(-2, -1, 4), rng.uniform(1, 2, 4)])
        at = np.ix_(g + groups * np.arange(8), g + groups * np.arange(8))
        H[at] = (Q * w) @ Q.T
        D[at] = Q[:, :4] @ Q[:, :4].T
    Dt = torch.empty(n, n, dtype=torch.float64, device="cuda")
    solver = DensitySolver(ctx, n, sp2_opts("tf32x3", max_iter=60, tau=1e-300))
    solver(torch.as_tensor(H, device="cuda"), 4.0 * groups, Dt)
    torch.cuda.synchronize()
    rep = report_to_dict(solver.report)
    assert rep["status"] == tbmd.TB_OK
    # eigenvalues one away from the chemical potential: FP32 rounding of the products only,
    # the bound of the vanishing threshold on a water system
    assert np.linalg.norm(Dt.cpu().numpy() - D) / np.sqrt(n) < 3e-6
    nsb = (n + 127) // 128
    pad = np.zeros((nsb * 128, nsb * 128))
    pad[:n, :n] = np.abs(H)
    live = (pad.reshape(nsb, 128, nsb, 128).max(axis=(1, 3)) > 0).astype(np.int64)
    assert rep["block_products"] == rep["iters"] * int((live @ live).sum())
