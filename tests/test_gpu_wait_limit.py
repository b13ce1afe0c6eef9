"""Short pipeline wait limits on the single-launch chains: a call either says TB_ERR_TIMEOUT or
has done all of its work, whichever of its thread blocks gave up, and the context stays usable."""

import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import (DensitySolver, FermiSolver, fermi_opts, fermi_report_to_dict,
                                          report_to_dict, sp2_opts)
from workloads import random_gapped_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n", [("fermi", 100), ("fermi", 700), ("sp2", 100), ("sp2", 700)])
def test_a_call_that_says_ok_is_complete(ctx, kind, n):
    H, _ = random_gapped_matrix(n, n // 2, gap=2.0, width=20.0, seed=n)
    Ht = torch.as_tensor(H, device="cuda")
    if kind == "fermi":
        s = FermiSolver(ctx, n, fermi_opts())
    else:
        s = DensitySolver(ctx, n, sp2_opts("tf32x3"))

    def call():
        D = torch.full_like(Ht, float("nan"))
        if kind == "fermi":
            s.mu.fill_(float("nan"))
            s(Ht, float(n // 2), 0.3, D)
            torch.cuda.synchronize()
            return D, fermi_report_to_dict(s.report)["status"]
        s(Ht, float(n // 2), D)
        torch.cuda.synchronize()
        return D, report_to_dict(s.report)["status"]

    D0, status = call()
    assert status == tbmd.TB_OK
    try:
        for limit in (1, 1000, 2000, 4000, 8000, 16000, 32000, 64000, 128000, 1000000000):
            for _ in range(5):
                tbmd.tb_ctx_set_wait_limit(ctx, limit)
                D, status = call()
                assert status in (tbmd.TB_OK, tbmd.TB_ERR_TIMEOUT)
                assert status == tbmd.TB_ERR_TIMEOUT or torch.equal(D, D0), limit
                assert limit > 1 or status == tbmd.TB_ERR_TIMEOUT
                assert limit < 1000000000 or status == tbmd.TB_OK
    finally:
        tbmd.tb_ctx_set_wait_limit(ctx, 2_000_000_000)
    D, status = call()
    assert status == tbmd.TB_OK and torch.equal(D, D0)


def test_the_limit_does_not_count_other_products(ctx):
    """n = 1500: a product takes about 50 us, its pipeline waits a few.  Warps that take part in
    some products only wait for several in between; a limit of 100 us is not theirs."""
    n = 1500
    H, _ = random_gapped_matrix(n, n // 2, gap=2.0, width=20.0, seed=n)
    Ht = torch.as_tensor(H, device="cuda")
    s = FermiSolver(ctx, n, fermi_opts())
    out = []
    for limit in (2_000_000_000, 100_000):
        D = torch.full_like(Ht, float("nan"))
        s.mu.fill_(float("nan"))
        tbmd.tb_ctx_set_wait_limit(ctx, limit)
        try:
            s(Ht, float(n // 2), 0.3, D)
            torch.cuda.synchronize()
        finally:
            tbmd.tb_ctx_set_wait_limit(ctx, 2_000_000_000)
        assert fermi_report_to_dict(s.report)["status"] == tbmd.TB_OK, limit
        out.append(D)
    assert torch.equal(out[0], out[1])
