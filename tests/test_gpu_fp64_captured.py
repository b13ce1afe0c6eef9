"""Captured FP64 SP2 calls around the sizes where their units no longer fit half the chip, or a
whole round of it: the eager call's D to the last bit, alone and several at once."""

import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import DensitySolver, report_to_dict, sp2_opts
from workloads import random_gapped_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [96, 104, 136, 176, 192, 272, 512])
def test_captured_calls_at_once(ctx, n):
    runs = []
    for k in range(5):
        H, _ = random_gapped_matrix(n, n // 2, gap=2.0, width=20.0, seed=10 * n + k)
        Ht = torch.as_tensor(H, device="cuda")
        D0, D = torch.empty_like(Ht), torch.empty_like(Ht)
        s = DensitySolver(ctx, n, sp2_opts("fp64", tol=1e-11))
        s(Ht, float(n // 2), D0)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            s(Ht, float(n // 2), D)
        runs.append((Ht, D0, D, s, g, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(4):
        for _, _, _, _, g, st in runs:
            with torch.cuda.stream(st):
                g.replay()
    torch.cuda.synchronize()
    for _, D0, D, s, _, _ in runs:
        assert report_to_dict(s.report)["status"] == tbmd.TB_OK
        assert torch.equal(D, D0)
