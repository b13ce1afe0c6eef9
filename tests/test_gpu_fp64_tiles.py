"""The launched FP64 products on both sides of the rule that leaves out the lower tiles (more tiles
than SMs): D against the eigenvalue projector, exactly symmetric, and the report's traces, which
count mirrored tiles twice."""

import numpy as np
import pytest
import torch

from oracle import density
from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import DensitySolver, report_to_dict, sp2_opts
from workloads import random_gapped_matrix

pytestmark = pytest.mark.gpu


# 64 x 64 tiles: 81, 144 and 169 of them; launch timing selects the launched form below n = 513
# (16 x 16 tiles: 9, 144 and 169)
@pytest.mark.parametrize("n,timed", [(513, False), (768, False), (769, False), (48, True), (192, True), (193, True)])
def test_launched_fp64(ctx, n, timed):
    H, _ = random_gapped_matrix(n, n // 3, gap=2.0, width=20.0, seed=n)
    Ht = torch.as_tensor(H, device="cuda")
    D = torch.full_like(Ht, float("nan"))
    s = DensitySolver(ctx, n, sp2_opts("fp64", tol=1e-11))
    tbmd.tb_ctx_set_profiling(ctx, timed)
    try:
        s(Ht, float(n // 3), D)
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_profiling(ctx, False)
    r = report_to_dict(s.report)
    assert r["status"] == tbmd.TB_OK
    assert torch.equal(D, D.T.contiguous())
    D = D.cpu().numpy()
    # the bound of the same comparison in test_gpu_run.py
    assert np.linalg.norm(D - density.density_T0(H, n // 3).D) / np.sqrt(n) < 1e-9
    # FP64 sums of n and n^2 terms of magnitude one at most
    assert abs(r["trace"] - np.trace(D)) < 1e-13 * n
    assert abs(r["trace"] - r["idem_trace"] - (D ** 2).sum()) < 1e-12 * n
