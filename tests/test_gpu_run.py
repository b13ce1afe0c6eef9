"""The single-launch forms of dm_fermi and of dm_sp2's tensor-core phase: tile
edges, every unit width, cut last rounds, one cluster and a cooperative grid."""

import numpy as np
import pytest
import torch

from oracle import density
from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import (DensitySolver, FermiSolver, fermi_opts, fermi_report_to_dict,
                                          report_to_dict, sp2_opts)
from workloads import random_gapped_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = tbmd.Context()
    yield c
    c.close()


def _banded(n, seed):
    """A symmetric matrix with a 2 eV gap in its middle and a spectral width of ~14 eV."""
    rng = np.random.default_rng(seed)
    H = np.diag(np.where(np.arange(n) < n // 2, -4.0, 4.0) + rng.uniform(-1, 1, n))
    for k in (1, 2, 5):
        if k < n:
            H += np.diag(rng.uniform(-0.3, 0.3, n - k), k) + 0.0
    return np.triu(H) + np.triu(H, 1).T


# n: one CTA; a ragged tile; the cluster's edges (ld 640 / 768); 32-, 64- and 128-column
# units on the whole chip; grid limits that give several rounds, and last rounds cut in 2 and 4
@pytest.mark.parametrize("n,limit", [(1, 0), (2, 0), (31, 0), (128, 0), (129, 0), (300, 0), (640, 0), (641, 0),
                                     (1100, 0), (1600, 0), (300, 1), (300, 5), (400, 8), (513, 12)])
def test_fermi_single_launch(ctx, n, limit):
    H = _banded(n, n)
    nocc, kT = 0.5 * n - (0.25 if n < 3 else 0.0), 0.15
    Ht = torch.as_tensor(H, device="cuda")
    D = torch.full_like(Ht, float("nan"))
    s = FermiSolver(ctx, n, fermi_opts())
    tbmd.tb_ctx_set_grid_limit(ctx, limit)
    try:
        s(Ht, nocc, kT, D)
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_grid_limit(ctx, 0)
    rep = fermi_report_to_dict(s.report)
    assert rep["status"] == tbmd.TB_OK
    Dn = D.cpu().numpy()
    assert np.array_equal(Dn, Dn.T)
    # dm_fermi's bound: FP32-level products whose errors add up over the doubling steps
    assert np.linalg.norm(Dn - density.density_fermi(H, nocc, kT).D) / np.sqrt(n) < 2e-6


@pytest.mark.parametrize("n", [1, 127, 130, 300, 640, 700, 1300, 1700])
@pytest.mark.parametrize("prec", ["tf32", "tf32x3"])
def test_sp2_single_launch_is_the_launched_form(ctx, n, prec):
    """Same products, same order: the same D to the last bit, eagerly and captured (launch
    timing selects the launched form)."""
    H = _banded(n, n + 1)
    nocc = float(n // 2)
    Ht = torch.as_tensor(H, device="cuda")
    s = DensitySolver(ctx, n, sp2_opts(prec, refine=0 if n > 1500 else 2))
    out = []
    for form in ("launched", "single", "captured"):
        D = torch.full_like(Ht, float("nan"))
        tbmd.tb_ctx_set_profiling(ctx, form == "launched")
        if form == "captured":
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, capture_error_mode="thread_local"):
                s(Ht, nocc, D)
            for _ in range(2):
                g.replay()
        else:
            s(Ht, nocc, D)
        torch.cuda.synchronize()
        out.append((D, report_to_dict(s.report)))
    tbmd.tb_ctx_set_profiling(ctx, False)
    (D0, r0), rest = out[0], out[1:]
    for D, r in rest:
        assert torch.equal(D, D0)
        for k in ("status", "iters", "refine_iters", "branches", "refine_branches", "eps_min", "eps_max"):
            assert r[k] == r0[k]
        assert abs(r["trace"] - r0["trace"]) <= 1e-12 * max(1.0, n)


@pytest.mark.parametrize("limit", [1, 4, 7, 24])
def test_sp2_single_launch_on_few_ctas(ctx, limit):
    H, _ = random_gapped_matrix(600, 250, gap=4.0, width=20.0, seed=3)
    Ht = torch.as_tensor(H, device="cuda")
    s = DensitySolver(ctx, 600, sp2_opts("tf32x3", refine=0))
    D0, D = torch.empty_like(Ht), torch.empty_like(Ht)
    s(Ht, 250.0, D0)
    tbmd.tb_ctx_set_grid_limit(ctx, limit)
    try:
        s(Ht, 250.0, D)
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_grid_limit(ctx, 0)
    assert torch.equal(D, D0)
    assert report_to_dict(s.report)["status"] == tbmd.TB_OK


def test_two_streams_at_once(ctx):
    """Calls on two streams with workspaces of their own do not disturb each other."""
    sizes, res = (900, 1000), []
    Hs = [torch.as_tensor(_banded(n, n), device="cuda") for n in sizes]
    sol = [FermiSolver(ctx, n, fermi_opts()) for n in sizes]
    Ds = [torch.empty_like(H) for H in Hs]
    for s, H, D, n in zip(sol, Hs, Ds, sizes):
        s(H, 0.5 * n, 0.2, D)
        torch.cuda.synchronize()
        res.append(D.clone())
        s.mu.fill_(float("nan"))
    streams = [torch.cuda.Stream() for _ in sizes]
    torch.cuda.synchronize()
    for _ in range(3):
        for s, H, D, n, st in zip(sol, Hs, Ds, sizes, streams):
            with torch.cuda.stream(st):
                s.mu.fill_(float("nan"))
            s(H, 0.5 * n, 0.2, D, stream=st)
    torch.cuda.synchronize()
    for s, D, R in zip(sol, Ds, res):
        assert fermi_report_to_dict(s.report)["status"] == tbmd.TB_OK
        assert torch.equal(D, R)


# units of 8 x 8 (to n = 136) and 16 x 16; one cluster, one unit per SM, several; grid limits
@pytest.mark.parametrize("n,limit", [(1, 0), (7, 0), (8, 0), (40, 0), (48, 0), (48, 3), (136, 0), (137, 0), (200, 16),
                                     (300, 0), (512, 0), (513, 0)])
def test_fp64_single_launch(ctx, n, limit):
    """The FP64 recursion against the eigenvalue projector and against the launched form (same
    branches; sums over K in another order: a rounding of 1e-16 n per product, which the
    projections of converged eigenvalues contract)."""
    H = _banded(n, n + 2)
    nocc = float(n // 2)
    Ht = torch.as_tensor(H, device="cuda")
    s = DensitySolver(ctx, n, sp2_opts("fp64", tol=1e-11))
    D0, D = torch.empty_like(Ht), torch.full_like(Ht, float("nan"))
    tbmd.tb_ctx_set_profiling(ctx, True)  # selects the launched form
    s(Ht, nocc, D0)
    torch.cuda.synchronize()
    r0 = report_to_dict(s.report)
    tbmd.tb_ctx_set_profiling(ctx, False)
    tbmd.tb_ctx_set_grid_limit(ctx, limit)
    try:
        s(Ht, nocc, D)
        g = torch.cuda.CUDAGraph()
        Dg = torch.empty_like(D)
        torch.cuda.synchronize()
        r = report_to_dict(s.report)
        with torch.cuda.graph(g, capture_error_mode="thread_local"):
            s(Ht, nocc, Dg)
        g.replay()
        torch.cuda.synchronize()
    finally:
        tbmd.tb_ctx_set_grid_limit(ctx, 0)
    assert r["status"] == r0["status"] == tbmd.TB_OK
    assert r["iters"] == r0["iters"] and r["branches"] == r0["branches"]
    assert torch.equal(Dg, D)
    assert (D - D0).abs().max().item() < 1e-12
    if 1 < n:
        assert np.linalg.norm(D.cpu().numpy() - density.density_T0(H, int(nocc)).D) / np.sqrt(n) < 1e-9
