"""A product that takes longer than the 2 s after which the waits between the products of a
single-launch chain give up: one CTA for a matrix of 7875 tiles (3 s), as a limit on the grid or a
matrix of n = 80 000 on the whole chip makes it."""

import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import DensitySolver, report_to_dict, sp2_opts

pytestmark = pytest.mark.gpu


def test_one_projection_of_seconds(ctx):
    n = 16000
    g = torch.Generator(device="cuda").manual_seed(1)
    H = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g).mul_(0.01)
    H = (H + H.T).contiguous()
    H.diagonal().add_(torch.linspace(-5.0, 5.0, n, dtype=torch.float64, device="cuda"))
    s = DensitySolver(ctx, n, sp2_opts("tf32x3", max_iter=1, refine=0))
    D0, D = torch.empty_like(H), torch.full_like(H, float("nan"))
    s(H, 0.5 * n, D0)
    torch.cuda.synchronize()
    r0 = report_to_dict(s.report)
    tbmd.tb_ctx_set_grid_limit(ctx, 1)
    try:
        s(H, 0.5 * n, D)
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_grid_limit(ctx, 0)
    r = report_to_dict(s.report)
    assert r["status"] == r0["status"] != tbmd.TB_ERR_TIMEOUT and r["iters"] == r0["iters"] == 1
    assert torch.equal(D, D0)
