"""Single-launch chains on a cluster that holds more CTAs than the matrix has units (clusters
are powers of two): the CTAs without units take no part, and every one of many calls gives the
same status and the same bits."""

import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import (DensitySolver, FermiSolver, fermi_opts, fermi_report_to_dict,
                                          report_to_dict, sp2_opts)
from workloads import random_gapped_matrix

pytestmark = pytest.mark.gpu


# tensor-core chains: 12 units on 16 CTAs (n = 200; captured also n = 300, 64 columns), 10 and 15
# tiles on 16 (captured, n = 500 and 600); FP64: 3 units on 4 CTAs, 6 on 8, 10 and 15 on 16
@pytest.mark.parametrize("kind,n,captured", [("sp2", 200, False), ("sp2", 300, True), ("sp2", 500, True),
                                             ("sp2", 600, True), ("fermi", 200, False), ("fermi", 300, True),
                                             ("fermi", 600, True), ("fp64", 16, False), ("fp64", 20, False),
                                             ("fp64", 32, True), ("fp64", 40, False)])
def test_chains_with_idle_ctas(ctx, kind, n, captured):
    H, _ = random_gapped_matrix(n, n // 2, gap=2.0, width=20.0, seed=n)
    Ht = torch.as_tensor(H, device="cuda")
    D = torch.full_like(Ht, float("nan"))
    if kind == "fermi":
        s = FermiSolver(ctx, n, fermi_opts())
        call, status = (lambda: s(Ht, float(n // 2), 0.3, D)), (lambda: fermi_report_to_dict(s.report)["status"])
    else:
        s = DensitySolver(ctx, n, sp2_opts("fp64", tol=1e-11) if kind == "fp64" else sp2_opts("tf32x3"))
        call, status = (lambda: s(Ht, float(n // 2), D)), (lambda: report_to_dict(s.report)["status"])
    if captured:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            call()
        call = g.replay
    first = None
    for _ in range(100):
        if kind == "fermi":
            s.mu.fill_(float("nan"))
        call()
        torch.cuda.synchronize()
        assert status() == tbmd.TB_OK
        first = D.clone() if first is None else first
        assert torch.equal(D, first)
    if kind != "fermi":  # the launched form, which launch timing selects: the same products
        tbmd.tb_ctx_set_profiling(ctx, True)
        try:
            s(Ht, float(n // 2), D)
            torch.cuda.synchronize()
        finally:
            tbmd.tb_ctx_set_profiling(ctx, False)
        # FP64: sums over K in another order (1e-16 n a product, which the projections contract)
        assert (D - first).abs().max().item() <= (1e-12 if kind == "fp64" else 0.0)
