"""dm_fermi's single-launch form (tf32, tf32x3) against its launched form, bit by bit, and
against itself on workspaces full of NaN: nothing is read before it is written.

One expansion at a given mu with the electron count far away: no shift of the chemical
potential follows, so D depends on the products alone (the FP64 trace sums of the two forms
differ in order).  A gapless spectrum keeps every product's rounding visible in D; a gap would
contract it."""

import numpy as np
import pytest
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import FermiSolver, fermi_opts, fermi_report_to_dict

pytestmark = pytest.mark.gpu
KT = 0.5


@pytest.fixture(scope="module")
def ctx():
    c = tbmd.Context()
    yield c
    c.close()


def _gapless(n, seed):
    A = torch.as_tensor(np.random.default_rng(seed).normal(0.0, 3.0 / np.sqrt(n), (n, n)), device="cuda")
    return 0.5 * (A + A.T).contiguous()


def _call(ctx, s, H, nocc, limit=0, captured=False):
    """D of one call on a workspace whose every word is a NaN."""
    D = torch.full_like(H, float("nan"))
    s.ws.buf.fill_(0xFF)
    s.mu.fill_(float("nan"))
    torch.cuda.synchronize()
    tbmd.tb_ctx_set_grid_limit(ctx, limit)
    try:
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, capture_error_mode="thread_local"):
                s(H, nocc, KT, D)
            g.replay()
        else:
            s(H, nocc, KT, D)
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_grid_limit(ctx, 0)
    return D, fermi_report_to_dict(s.report)


# n and the grid limits of the single-launch form (0: the whole chip): one 32-, 64- and
# 128-column unit a CTA, several units a CTA, a last round cut in two and in four
@pytest.mark.parametrize("n,limits", [(300, (0, 4, 5)), (700, (0, 13, 20)), (1100, (0, 40)), (1500, (0,)),
                                      (2400, (0,))])
@pytest.mark.parametrize("prec", ["tf32", "tf32x3"])
def test_one_expansion_is_the_launched_form(ctx, n, limits, prec):
    H = _gapless(n, n)
    s = FermiSolver(ctx, n, fermi_opts(prec, mu_iters=1))
    # captured on fewer CTAs than the matrix has tiles: the launched form
    D0, r0 = _call(ctx, s, H, 0.3 * n, limit=4, captured=True)
    assert bool(torch.isfinite(D0).all())
    assert r0["status"] == tbmd.TB_ERR_NOT_CONVERGED and r0["mu_iters"] == 1
    for limit in limits:
        D, r = _call(ctx, s, H, 0.3 * n, limit)
        assert torch.equal(D, D0), limit
        assert r["status"] == r0["status"] and r["m"] == r0["m"] and r["mu"] == r0["mu"]
        assert abs(r["trace"] - r0["trace"]) <= 1e-12 * n  # FP64 sums of n terms below 1


@pytest.mark.parametrize("n", [60, 700, 900])
@pytest.mark.parametrize("prec", ["tf32", "tf32x3"])
def test_repeated_calls_agree(ctx, n, prec):
    """All expansions of a call, eagerly and captured: the same D each time."""
    H = _gapless(n, n + 1)
    s = FermiSolver(ctx, n, fermi_opts(prec))
    D0, r0 = _call(ctx, s, H, 0.3 * n)
    assert bool(torch.isfinite(D0).all()) and r0["mu_iters"] > 1
    for _ in range(10):
        assert torch.equal(_call(ctx, s, H, 0.3 * n)[0], D0)
    for _ in range(3):
        assert torch.equal(_call(ctx, s, H, 0.3 * n, captured=True)[0], D0)


def test_two_chains_share_the_chip(ctx):
    """Two cooperative grids of 36 CTAs (one tile each), which run at the same time: each call's D
    is the one it has alone."""
    sizes = (900, 1000)
    Hs = [_gapless(n, n + 2) for n in sizes]
    sol = [FermiSolver(ctx, n, fermi_opts()) for n in sizes]
    D0 = [_call(ctx, s, H, 0.3 * n, 60)[0] for s, H, n in zip(sol, Hs, sizes)]
    Ds = [torch.full_like(H, float("nan")) for H in Hs]
    streams = [torch.cuda.Stream() for _ in sizes]
    torch.cuda.synchronize()
    tbmd.tb_ctx_set_grid_limit(ctx, 60)
    try:
        for _ in range(10):
            for s, H, D, n, st in zip(sol, Hs, Ds, sizes, streams):
                with torch.cuda.stream(st):
                    s.mu.fill_(float("nan"))
                s(H, 0.3 * n, KT, D, stream=st)
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_grid_limit(ctx, 0)
    for s, D, R in zip(sol, Ds, D0):
        assert fermi_report_to_dict(s.report)["status"] == tbmd.TB_OK
        assert torch.equal(D, R)
