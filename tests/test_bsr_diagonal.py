"""Diagonal blocks of the block-sparse products of two matrices, which the epilogue makes
symmetric through a warp's shared-memory tile: the order of its accesses, from the source, and
repeated expansions on the GPU, bit by bit."""

import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_6836_gb300", "csrc")


def test_the_tile_is_free_before_a_lane_writes_another_layout():
    """tile_turn_in reads the tile lane by lane at a pitch of 128 bytes and tile_store across the
    lanes; the write at the tile's own pitch touches other lanes' values, so the warp has to meet
    in between."""
    with open(os.path.join(CSRC, "bsr.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    kernel = src[src.index("k_bsr_step_tc("):]
    write = kernel.index("s_sym[q][lane][j] = y[j]")
    before = max(kernel.rindex("tile_turn_in", 0, write), kernel.rindex("if (symd && c == q)", 0, write))
    assert "__syncwarp()" in kernel[before:write]


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
def test_repeated_expansions_agree(ctx, prec):
    """Products of two matrices with an S (E + E T, L - 4/3 L L^2) and without, several blocks a
    CTA's round: the same symmetric D from every call."""
    import torch

    from paper_1203_6836_gb300 import tbmd
    from paper_1203_6836_gb300.device import BsrMatrix, DeviceSystem, Workspace, fermi_opts, fermi_report_to_dict
    from workloads import ModelParams, water_system

    s = water_system(510, density=1.0, seed=4, morton=True)
    p = ModelParams()
    ds = DeviceSystem(s.R, s.types, s.box)
    n, nsb = ds.norb, (ds.norb + 127) // 128
    f64 = dict(dtype=torch.float64, device="cuda")
    Hb, Db = BsrMatrix(n, nsb * nsb), BsrMatrix(n, nsb * nsb)
    v = torch.zeros(ds.natoms, **f64)
    ws = Workspace(tbmd.tb_bsr_model_workspace_size(ds.natoms, n))
    tbmd.tb_build_H_bsr(ctx, tbmd.tb_params.from_model(p), ds.sys, ds.R, None, Hb.mat, v, ws.ptr, ws.nbytes)
    o = fermi_opts(prec)
    fws = Workspace(tbmd.dm_fermi_sparse_workspace_size(n, o, 0))
    rep = torch.zeros(128, dtype=torch.uint8, device="cuda")
    first = None
    for _ in range(20):
        mu = torch.full((1,), float("nan"), **f64)
        fws.buf.fill_(0xFF)
        tbmd.dm_fermi_sparse(ctx, Hb.mat, s.n_occ(p), 0.5, o, 1e-6, 0, Db.mat, mu, fws.ptr, fws.nbytes, rep)
        torch.cuda.synchronize()
        assert fermi_report_to_dict(rep)["status"] in (tbmd.TB_OK, tbmd.TB_ERR_NOT_CONVERGED)
        D = Db.to_dense()
        assert np.isfinite(D).all() and np.array_equal(D, D.T)
        first = D if first is None else first
        assert np.array_equal(D, first)
