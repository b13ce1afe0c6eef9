"""The closing kick on a cluster of eight blocks: its order of cluster barriers and accesses to
the first block's shared memory, from the source, and its sums on the GPU."""

import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_6836_gb300", "csrc")


def test_every_block_has_started_before_its_shared_memory_is_written():
    """A distributed shared-memory access needs a cluster barrier before it (the other block has
    started) and one after it (the other block has not left)."""
    with open(os.path.join(CSRC, "md.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    kernel = src[src.index("k_kick_energy("):src.index("int launch_kick_energy")]
    at = kernel.index("map_shared_rank")
    assert "this_cluster().sync()" in kernel[:at]
    assert "this_cluster().sync()" in kernel[at:]


@pytest.mark.gpu
@pytest.mark.parametrize("molecules", [171, 500, 683])
def test_kinetic_energy_on_a_cluster(ctx, molecules):
    """513, 1500 and 2049 atoms: kinetic energy and max|n - q| of each of several steps."""
    import torch

    from oracle import observables
    from paper_1203_6836_gb300 import tbmd
    from paper_1203_6836_gb300.device import DeviceSystem, MDState, sp2_opts, xl_params
    from workloads import XLParams, gapped_params, gapped_vapour, thermal_velocities

    p = gapped_params()
    s = gapped_vapour(molecules, seed=1)
    M = s.masses(p)
    opts = sp2_opts("tf32x3", max_iter=100, refine=2)
    xl = XLParams()
    st = MDState(DeviceSystem(s.R, s.types, s.box), thermal_velocities(M, 300.0, seed=2), M, s.n_occ(p), xl.K, opts)
    xp = xl_params(xl.dt, xl.kappa, xl.alpha, xl.c)
    tp = tbmd.tb_params.from_model(p)
    tbmd.xlbomd_init(ctx, tp, st.st, xp, opts, 1e-6, 100)
    for k in range(1, 6):
        tbmd.xlbomd_step(ctx, tp, st.st, xp, opts)
        torch.cuda.synchronize()
        e = st.energies.cpu().numpy()
        # FP64 sums of at most 2049 positive terms on both sides
        assert e[5] == pytest.approx(observables.kinetic_energy(st.v.cpu().numpy(), M), rel=1e-12)
        assert e[6] == (st.n_hist[0] - st.q).abs().max().item()  # no rounding: a maximum
        assert e[7] == k and np.isfinite(e).all()
