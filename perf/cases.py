"""What is timed: the calls that a program built on this library makes, from one 24-atom step to
the block-sparse steps of 16 383 atoms and a served mix of trajectories.

Every case builds seeded water-like inputs (plain positions and charges; nothing of the method's
own arithmetic) and goes through the package's public entry points.  `exact` restates the model
in 64-bit torch and diagonalises, with none of the package's code.

Units: eV, Angstrom, amu, fs.
"""

import itertools
import math

import numpy as np
import torch

from paper_1203_6836_gb300 import tbmd
from paper_1203_6836_gb300.device import (BsrMatrix, DensitySolver, DeviceSystem, FermiSolver, MDState, Server,
                                          Workspace, fermi_opts, new_report, sp2_opts, xl_params)

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)

# model constants of the three recipes the tests and the benchmark use
PLAIN = dict(eps_s_O=-20.0, eps_p_O=-12.0, eps_s_H=-7.0, t_hop=3.0, r_decay=0.5, hubbard_u=10.0, coulomb_k=14.399645,
             gamma_cut=6.0, r1=5.0, rcut=6.0, n0_O=6.0, n0_H=1.0, pair_a=24.0, pair_rho=0.3, zeta_a2=0.0, zeta_a3=0.0,
             zeta_a4=0.0, pair_a2=0.0, pair_a3=0.0, pair_a4=0.0, gamma_form=0, ewald_alpha=0.0, overlap_s0=0.0,
             overlap_rs=0.4)
GAPPED = dict(PLAIN, t_hop=20.0, r_decay=0.4, hubbard_u=6.0, pair_a=65.75)
OVERLAP = dict(GAPPED, overlap_s0=1.1, pair_a=24.14)

# integrator: K = 5, kappa = kappa0 / 2
DT, KAPPA, ALPHA, CK = 0.25, 0.91, 0.018, (-6.0, 14.0, -8.0, -3.0, 4.0, -1.0)
ACC = 9.648533e-3  # 1 eV / (A amu) in A / fs^2
AMU_G = 1.66054    # 1 amu in 1e-24 g
KB = 8.617333262e-5


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # one step of the paper's method in 64 bits on 8 molecules: launches and latency only
        {"name": "md_24_fp64", "kind": "md", "molecules": 8, "precision": "fp64", "refine": 0, "graph": False},
        # the T = 0 density matrix of a 300-atom liquid, a usual size of an ab-initio-style run
        {"name": "sp2_300", "kind": "sp2", "atoms": 300, "precision": "tf32x3", "refine": 2},
        # the same for the 2048-atom system the benchmark is quoted on
        {"name": "sp2_2048", "kind": "sp2", "atoms": 2048, "precision": "tf32x3", "refine": 2},
        # a whole step of T = 0 dynamics on 2046 atoms
        {"name": "md_2046", "kind": "md", "molecules": 682, "precision": "tf32x3", "refine": 2, "graph": False},
        # finite-temperature density matrices, chemical potential known from the step before: a small
        # trajectory of the served mix, and a large one
        {"name": "fermi_96", "kind": "fermi", "molecules": 32, "kT": 0.1},
        {"name": "fermi_1200", "kind": "fermi", "molecules": 400, "kT": 0.1},
        # many independent small systems, 16 to 256 atoms each, in one launch
        {"name": "batch_512", "kind": "batch", "count": 512, "lo": 16, "hi": 256},
        # thresholded density matrix of a dense liquid, a quarter of the 16384-atom workload
        {"name": "bsr_liquid_4096", "kind": "bsr_sp2", "atoms": 4096},
        # linear-scaling dynamics: one block-sparse step of 16383 atoms of vapour
        {"name": "bsr_md_16383", "kind": "bsr_md", "molecules": 5461},
        # the finite-temperature density matrix of the same
        {"name": "bsr_fermi_16383", "kind": "bsr_fermi", "molecules": 5461, "kT": 0.2},
        # a step in a non-orthogonal basis
        {"name": "nonorth_192", "kind": "nonorth", "molecules": 64, "precision": "tf32x3", "refine": 2},
        # one step of each of 12 trajectories of uneven size through the step server, read back
        {"name": "serve_12", "kind": "serve", "trajectories": 12, "lo": 32, "hi": 600},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["md", "sp2", "fermi", "batch", "bsr_sp2", "bsr_md", "bsr_fermi", "nonorth", "serve"])
    if kind == "md":
        m = size(8, 682)
        fp64 = m <= 64 and rng.random() < 0.7
        return {"kind": kind, "molecules": m, "precision": "fp64" if fp64 else "tf32x3", "refine": 0 if fp64 else 2,
                "graph": rng.random() < 0.5}
    if kind == "sp2":
        return {"kind": kind, "atoms": size(24, 2048), "precision": rng.choice(["tf32x3", "tf32x3", "bf16x3"]),
                "refine": rng.choice([1, 2, 3])}
    if kind == "fermi":
        return {"kind": kind, "molecules": size(11, 400), "kT": rng.choice([0.1, 0.2, 0.5])}
    if kind == "batch":
        lo = rng.randint(16, 64)
        return {"kind": kind, "count": size(32, 512), "lo": lo, "hi": rng.randint(lo + 1, 256)}
    if kind == "bsr_sp2":
        return {"kind": kind, "atoms": size(600, 4096)}
    if kind in ("bsr_md", "bsr_fermi"):
        c = {"kind": kind, "molecules": size(400, 5461)}
        return dict(c, kT=rng.choice([0.2, 0.3])) if kind == "bsr_fermi" else c
    if kind == "nonorth":
        return {"kind": kind, "molecules": size(8, 64), "precision": rng.choice(["tf32x3", "fp64"]), "refine": 2}
    return {"kind": kind, "trajectories": rng.randint(3, 12), "lo": 32, "hi": rng.randint(64, 600)}


# ---------------------------------------------------------------- seeded inputs

def _box(n_O, n_H, density):
    return ((16.0 * n_O + n_H) * AMU_G / density) ** (1.0 / 3.0)


def _morton(R, box, cell=3.0):
    m = max(1, int(box // cell))
    ijk = np.minimum((R / box * m).astype(np.int64), m - 1)
    code = np.zeros(len(R), dtype=np.int64)
    for bit in range(21):
        for ax in range(3):
            code |= ((ijk[:, ax] >> bit) & 1) << (3 * bit + ax)
    return np.argsort(code, kind="stable")


def liquid(atoms, seed, morton=False):
    """Water-like liquid at 1.0 g/cc: atoms at random sites of a cubic grid, displaced so that
    no two come closer than 0.9 A; a third O-like, an even number of H-like."""
    rng = np.random.default_rng(seed)
    n_O = atoms // 3
    if (atoms - n_O) % 2:
        n_O -= 1
    n_H = atoms - n_O
    box = _box(n_O, n_H, 1.0)
    m = 1
    while m ** 3 < atoms:
        m += 1
    a = box / m
    site = rng.permutation(m ** 3)[:atoms]
    ijk = np.stack([site // (m * m), (site // m) % m, site % m], 1)
    R = np.mod((ijk + 0.5) * a + rng.uniform(-1, 1, (atoms, 3)) * max(0.0, (a - 0.9) / 2), box)
    types = np.array([tbmd.TB_TYPE_O] * n_O + [tbmd.TB_TYPE_H] * n_H, dtype=np.int32)
    if morton:
        o = _morton(R, box)
        R, types = R[o], types[o]
    return np.ascontiguousarray(R), np.ascontiguousarray(types), box


def vapour(molecules, seed, morton=False):
    """H2O-like molecules (O-H 0.96 A, 104.5 degrees) at 0.1 g/cc on a jittered cubic grid,
    randomly turned; all O first, or in Morton order."""
    rng = np.random.default_rng(seed)
    box = _box(molecules, 2 * molecules, 0.1)
    m = 1
    while m ** 3 < molecules:
        m += 1
    k = np.arange(molecules)
    O = (np.stack([k // (m * m), (k // m) % m, k % m], 1) + 0.5) / m * box + rng.normal(0, 0.1, (molecules, 3))
    Q = np.linalg.qr(rng.standard_normal((molecules, 3, 3)))[0]
    t = math.radians(104.5) / 2
    u = 0.96 * np.array([[math.sin(t), math.cos(t), 0.0], [-math.sin(t), math.cos(t), 0.0]])
    Hs = O[:, None, :] + np.einsum("mij,hj->mhi", Q, u)
    R = np.mod(np.concatenate([O, Hs.reshape(-1, 3)]), box)
    types = np.array([tbmd.TB_TYPE_O] * molecules + [tbmd.TB_TYPE_H] * (2 * molecules), dtype=np.int32)
    if morton:
        o = _morton(R, box)
        R, types = R[o], types[o]
    return np.ascontiguousarray(R), np.ascontiguousarray(types), box


def n_occ(types):
    n_O = int(np.count_nonzero(types == tbmd.TB_TYPE_O))
    return 0.5 * (6 * n_O + (len(types) - n_O))


def masses(types):
    return np.where(types == tbmd.TB_TYPE_O, 16.0, 1.0)


# charge of an O-like atom of a molecule at self-consistency, by recipe
Q_PLAIN, Q_GAPPED, Q_OVERLAP = 1.21, 1.30, 1.76


def charges(types, seed, o):
    """Charges as they are along a trajectory of such molecules: O-like `o` e, H-like -o/2, and
    what the neighbours change."""
    rng = np.random.default_rng(seed + 77)
    q = np.where(types == tbmd.TB_TYPE_O, o, -o / 2) + rng.normal(0, 0.02, len(types))
    return q - q.mean()


def checkpoint(types, seed, o):
    """What a step reads of its trajectory: velocities at 300 K, forces, the last charges, and
    the auxiliary charges of the last six steps (a slow drift)."""
    rng = np.random.default_rng(seed + 99)
    N, m = len(types), masses(types)
    v = rng.standard_normal((N, 3)) * np.sqrt(KB * 300.0 / m * ACC)[:, None]
    v -= (m[:, None] * v).sum(0) / m.sum()
    F = rng.normal(0, 0.3, (N, 3))
    n0, dn = charges(types, seed, o), rng.normal(0, 1e-3, N)
    dn -= dn.mean()
    hist = np.stack([n0 - k * dn for k in range(len(CK))])
    return v, F - F.mean(0), n0 + 0.5 * dn, hist


def batch_sizes(case):
    """Atom counts of a batch, spread over [lo, hi]: the same for every seed."""
    return np.random.default_rng(4).integers(case["lo"], case["hi"] + 1, size=case["count"])


def serve_sizes(case):
    """Molecules of the served trajectories, spread over the logarithm of [lo, hi] atoms."""
    x = np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["trajectories"])
    return [max(1, int(round(math.exp(v) / 3))) for v in x]


# ---------------------------------------------------------------- prepare

def params(p):
    return tbmd.tb_params(**p)


def hamiltonian(ctx, p, R, types, box, n):
    ds = DeviceSystem(R, types, box)
    H = torch.empty(ds.norb, ds.norb, **F64)
    G = torch.empty(ds.natoms, ds.natoms, **F64)
    tbmd.tb_build_H(ctx, params(p), ds.sys, ds.R, torch.as_tensor(n, device=DEV) if n is not None else None, H, G)
    return H


def prepare(case, seed):
    return globals()["prepare_" + case["kind"]](case, seed)


def run(state):
    return globals()["run_" + state["kind"]](state)


def prepare_sp2(case, seed):
    ctx = tbmd.Context()
    R, types, box = liquid(case["atoms"], seed)
    H = hamiltonian(ctx, PLAIN, R, types, box, None)
    solver = DensitySolver(ctx, H.shape[0], sp2_opts(case["precision"], max_iter=100, refine=case["refine"]))
    return {"kind": "sp2", "H": H, "n_occ": n_occ(types), "D": torch.empty_like(H), "solver": solver}


def run_sp2(s):
    return s["solver"](s["H"], s["n_occ"], s["D"])


def prepare_fermi(case, seed):
    ctx = tbmd.Context()
    R, types, box = vapour(case["molecules"], seed)
    H = hamiltonian(ctx, PLAIN, R, types, box, charges(types, seed, Q_PLAIN))
    solver = FermiSolver(ctx, H.shape[0], fermi_opts())
    D = torch.empty_like(H)
    # the chemical potential extrapolated from earlier steps: near, not exact
    solver(H, n_occ(types), case["kT"], D)
    return {"kind": "fermi", "H": H, "n_occ": n_occ(types), "kT": case["kT"], "D": D, "solver": solver,
            "mu": solver.mu + 0.002}


def run_fermi(s):
    s["solver"].mu.copy_(s["mu"])
    s["solver"](s["H"], s["n_occ"], s["kT"], s["D"])
    return {"D": s["D"], "mu": s["solver"].mu}


def prepare_batch(case, seed):
    ctx = tbmd.Context()
    sizes = batch_sizes(case)
    systems = [liquid(int(N), 1000 * seed + i) for i, N in enumerate(sizes)]
    ns = [int(np.where(t == tbmd.TB_TYPE_O, 4, 1).sum()) for _, t, _ in systems]
    flat_H = torch.empty(sum(n * n for n in ns), **F64)
    flat_D = torch.zeros_like(flat_H)
    Hs, Ds, o, tp = [], [], 0, params(PLAIN)
    for (R, types, box), n in zip(systems, ns):
        ds = DeviceSystem(R, types, box)
        Hs.append(flat_H[o:o + n * n])
        Ds.append(flat_D[o:o + n * n])
        tbmd.tb_build_H(ctx, tp, ds.sys, ds.R, None, Hs[-1], torch.empty(ds.natoms, ds.natoms, **F64))
        o += n * n
    opts = sp2_opts("tf32x3", max_iter=100, tol=1e-8)
    ws = Workspace(tbmd.dm_sp2_grouped_workspace_size(ns, opts))
    tbmd.dm_sp2_grouped_plan(ctx, ns, [n_occ(t) for _, t, _ in systems], Hs, Ds, None, opts, 0, ws.ptr, ws.nbytes)
    return {"kind": "batch", "ctx": ctx, "ws": ws, "H": flat_H, "D": flat_D}


def run_batch(s):
    tbmd.dm_sp2_grouped_run(s["ctx"], s["ws"].ptr)
    return s["D"]


def prepare_md(case, seed, p=GAPPED, nonorth=False, bsr=None):
    ctx = tbmd.Context()
    R, types, box = vapour(case["molecules"], seed, morton=bsr is not None)
    v, F, q, hist = checkpoint(types, seed, Q_OVERLAP if nonorth else Q_GAPPED)
    if bsr is not None:
        opts = sp2_opts("tf32x3", max_iter=40, tau=1e-5, blocks_per_row=bsr)
    else:
        opts = sp2_opts(case["precision"], max_iter=100, tol=1e-10, refine=case["refine"])
    ds = DeviceSystem(R, types, box)
    nsb = (ds.norb + 127) // 128
    st = MDState(ds, v, masses(types), n_occ(types), len(CK) - 1, opts, nonorth=nonorth,
                 bsr_cap=(min(64, nsb) * nsb, min(40, nsb) * nsb) if bsr is not None else None)
    st.F.copy_(torch.as_tensor(F))
    st.q.copy_(torch.as_tensor(q))
    st.n_hist.copy_(torch.as_tensor(hist))
    live = [st.R, st.v, st.F, st.q, st.n_hist, st.energies]
    s = {"kind": case["kind"], "ctx": ctx, "tp": params(p), "xp": xl_params(DT, KAPPA, ALPHA, CK), "opts": opts,
         "st": st, "live": live, "saved": [t.clone() for t in live], "graph": None}
    if case.get("graph"):
        tbmd.xlbomd_step(ctx, s["tp"], st.st, s["xp"], opts)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            tbmd.xlbomd_step(ctx, s["tp"], st.st, s["xp"], opts)
    return s


def run_md(s):
    """One step from the checkpoint (so that every pass is the same step)."""
    st = s["st"]
    torch._foreach_copy_(s["live"], s["saved"])
    if s["graph"] is not None:
        s["graph"].replay()
    else:
        tbmd.xlbomd_step(s["ctx"], s["tp"], st.st, s["xp"], s["opts"])
    out = {"R": st.R, "v": st.v, "F": st.F, "q": st.q, "n": st.n_hist, "E": st.energies}
    if st.bsr:
        return dict(out, D_rows=st.D_bsr.row_ptr, D_cols=st.D_bsr.col, D=st.D_bsr.val)
    return dict(out, D=st.D) if st.S is None else dict(out, D=st.D, W=st.W, S=st.S)


def prepare_nonorth(case, seed):
    return prepare_md(case, seed, OVERLAP, nonorth=True)


def prepare_bsr_md(case, seed):
    return prepare_md(case, seed, bsr=64)


run_nonorth = run_bsr_md = run_md


def bsr_hamiltonian(ctx, p, R, types, box, n, cap):
    ds = DeviceSystem(R, types, box)
    H = BsrMatrix(ds.norb, cap)
    ws = Workspace(tbmd.tb_bsr_model_workspace_size(ds.natoms, ds.norb))
    v = torch.empty(ds.natoms, **F64)
    tbmd.tb_build_H_bsr(ctx, params(p), ds.sys, ds.R, torch.as_tensor(n, device=DEV) if n is not None else None,
                        H.mat, v, ws.ptr, ws.nbytes)
    return ds, H


def prepare_bsr_sp2(case, seed):
    ctx = tbmd.Context()
    R, types, box = liquid(case["atoms"], seed, morton=True)
    nsb = (int(np.where(types == tbmd.TB_TYPE_O, 4, 1).sum()) + 127) // 128
    ds, H = bsr_hamiltonian(ctx, PLAIN, R, types, box, None, nsb * nsb)
    opts = sp2_opts("tf32x3", max_iter=60, tau=1e-5)
    return {"kind": "bsr_sp2", "ctx": ctx, "tp": params(PLAIN), "ds": ds, "H": H, "D": BsrMatrix(H.n, nsb * nsb),
            "n_occ": n_occ(types), "opts": opts, "ws": Workspace(tbmd.dm_sp2_workspace_size(H.n, opts)),
            "report": new_report(), "q": torch.empty(ds.natoms, **F64)}


def run_bsr_sp2(s):
    D = s["D"]
    tbmd.dm_sp2_sparse(s["ctx"], s["H"].mat, s["n_occ"], s["opts"], D.mat, s["ws"].ptr, s["ws"].nbytes, s["report"])
    tbmd.mulliken_bsr(s["ctx"], s["tp"], s["ds"].sys, D.mat, s["q"])
    return {"D_rows": D.row_ptr, "D_cols": D.col, "D": D.val, "q": s["q"]}


def prepare_bsr_fermi(case, seed):
    ctx = tbmd.Context()
    R, types, box = vapour(case["molecules"], seed, morton=True)
    nsb = (int(np.where(types == tbmd.TB_TYPE_O, 4, 1).sum()) + 127) // 128
    ds, H = bsr_hamiltonian(ctx, GAPPED, R, types, box, charges(types, seed, Q_GAPPED),
                            min(64, nsb) * nsb)
    opts, bpr = fermi_opts(), min(64, nsb)
    s = {"kind": "bsr_fermi", "ctx": ctx, "tp": params(GAPPED), "ds": ds, "H": H, "D": BsrMatrix(H.n, min(40, nsb) * nsb),
         "n_occ": n_occ(types), "kT": case["kT"], "opts": opts, "bpr": bpr,
         "ws": Workspace(tbmd.dm_fermi_sparse_workspace_size(H.n, opts, bpr)), "mu": torch.full((1,), math.nan, **F64),
         "q": torch.empty(ds.natoms, **F64)}
    fermi_sparse(s)
    s["mu0"] = s["mu"].clone()  # the chemical potential of the step before
    return s


def fermi_sparse(s):
    tbmd.dm_fermi_sparse(s["ctx"], s["H"].mat, s["n_occ"], s["kT"], s["opts"], 1e-5, s["bpr"], s["D"].mat, s["mu"],
                         s["ws"].ptr, s["ws"].nbytes)


def run_bsr_fermi(s):
    D = s["D"]
    s["mu"].copy_(s["mu0"])
    fermi_sparse(s)
    tbmd.mulliken_bsr(s["ctx"], s["tp"], s["ds"].sys, D.mat, s["q"])
    return {"D_rows": D.row_ptr, "D_cols": D.col, "D": D.val, "q": s["q"], "mu": s["mu"]}


def prepare_serve(case, seed):
    # kappa scaled as the served vapour needs; a rough start of the charges is enough for a step
    xp = xl_params(DT, 0.06 * 2 * KAPPA, ALPHA, CK)
    srv = Server(tbmd.Context(), params(PLAIN), xp, kT=0.1, max_slots=32, scf_tol=1e-2, scf_max_iter=6)
    for i, m in enumerate(serve_sizes(case)):
        R, types, box = vapour(m, 1000 * seed + i)
        srv.add(types, box, R, checkpoint(types, seed + i, Q_PLAIN)[0], masses(types), n_occ(types))
    return {"kind": "serve", "srv": srv}


def run_serve(s):
    srv = s["srv"]
    for t in range(len(srv.natoms)):
        srv.submit(t)
    srv.drain()
    return [srv.read(t) for t in range(len(srv.natoms))]


# ---------------------------------------------------------------- work

def orbitals(case):
    k = case["kind"]
    if k in ("sp2", "bsr_sp2"):
        n_O = case["atoms"] // 3
        n_O -= (case["atoms"] - n_O) % 2
        return case["atoms"] + 3 * n_O
    return 6 * case["molecules"]


def work(case):
    """Matrices in and out once; the symmetric products (n^3 operations each, the half that the
    symmetry leaves) of the projections or expansions that such inputs take."""
    k = case["kind"]
    if k == "batch":
        n3 = n2 = 0
        for N in batch_sizes(case):
            n = orbitals({"kind": "sp2", "atoms": int(N)})
            n3, n2 = n3 + float(n) ** 3, n2 + float(n) ** 2
        return {"bytes": 16 * n2, "flops": 30 * n3}
    if k == "serve":
        ns = [6.0 * m for m in serve_sizes(case)]
        return {"bytes": sum(16 * n * n for n in ns), "flops": sum(75 * n ** 3 for n in ns)}
    n = float(orbitals(case))
    if k in ("bsr_md", "bsr_fermi"):
        # about 8 blocks of 128 x 128 in a block row, and 60 products of blocks in one product
        rows = math.ceil(n / 128)
        products = 16 if k == "bsr_md" else 70
        return {"bytes": rows * 16.0 * 131072, "flops": products * rows * 30 * 2.0 * 128 ** 3}
    if k == "bsr_sp2":
        return {"bytes": 8.0 * n * n, "flops": 35 * n ** 3}
    if k == "fermi":
        return {"bytes": 16 * n * n, "flops": 70 * n ** 3}
    if k == "nonorth":
        return {"bytes": 40 * n * n, "flops": (20 + 25) * n ** 3}
    return {"bytes": 16 * n * n, "flops": (45 if k == "sp2" else 20) * n ** 3}


# ---------------------------------------------------------------- the same in 64 bits

def radial(a, rho, p):
    """a exp(-r / rho) up to r1, then the quintic that meets it there with two derivatives and
    vanishes with two at rcut."""
    f, D = a * math.exp(-p["r1"] / rho), p["rcut"] - p["r1"]
    A = np.array([[1, 0, 0, 0, 0, 0], [0, 1, 0, 0, 0, 0], [0, 0, 2, 0, 0, 0], [D ** k for k in range(6)],
                  [k * D ** max(k - 1, 0) for k in range(6)], [k * (k - 1) * D ** max(k - 2, 0) for k in range(6)]])
    B = np.linalg.solve(A, np.array([f, -f / rho, f / rho ** 2, 0, 0, 0]))

    def g(r):
        x = r - p["r1"]
        t = sum(float(b) * x ** k for k, b in enumerate(B))
        return torch.where(r < p["r1"], a * torch.exp(-r / rho), torch.where(r < p["rcut"], t, torch.zeros_like(r)))
    return g


def blocks(V, l):
    """Slater-Koster blocks [N, N, 4, 4] (s, px, py, pz) of radial values V and unit vectors l."""
    B = V.new_zeros(*V.shape, 4, 4)
    B[..., 0, 0] = -V
    B[..., 0, 1:] = V[..., None] * l
    B[..., 1:, 0] = -V[..., None] * l
    B[..., 1:, 1:] = V[..., None, None] * (2 * l[..., :, None] * l[..., None, :] - torch.eye(3, dtype=V.dtype, device=V.device))
    return B


class Exact:
    """The model of one system in 64 bits."""

    def __init__(self, R, types, box, p, device=None):
        self.p, self.box, self.types = p, box, types
        self.dev = torch.device(device or (DEV if torch.cuda.is_available() else "cpu"))
        comps = [(i, c) for i, t in enumerate(types) for c in range(4 if t == tbmd.TB_TYPE_O else 1)]
        self.atom = torch.tensor([a for a, _ in comps], device=self.dev)
        self.comp = torch.tensor([c for _, c in comps], device=self.dev)
        self.N, self.n = len(types), len(comps)
        isO = torch.as_tensor(types == tbmd.TB_TYPE_O, device=self.dev)
        self.n0 = torch.where(isO, p["n0_O"], p["n0_H"]).to(torch.float64)
        e = torch.where(isO[self.atom], torch.where(self.comp == 0, p["eps_s_O"], p["eps_p_O"]), p["eps_s_H"])
        self.onsite = e.to(torch.float64)
        self.n_occ = n_occ(types)
        self.build(torch.as_tensor(R, dtype=torch.float64, device=self.dev))

    def build(self, R):
        """h, gamma, S and E_pair of the positions R."""
        p, N = self.p, self.N
        eye = torch.eye(N, dtype=torch.float64, device=self.dev)
        d0 = R[None, :, :] - R[:, None, :]
        d0 = d0 - self.box * torch.round(d0.detach() / self.box)
        hop, phi = radial(p["t_hop"], p["r_decay"], p), radial(p["pair_a"], p["pair_rho"], p)
        ovl = radial(p["overlap_s0"], p["overlap_rs"], p)
        rc = max(p["rcut"], p["gamma_cut"])
        k = max(0, math.ceil(rc / self.box - 0.5))
        self.G = p["hubbard_u"] * eye
        self.E_pair = torch.zeros((), dtype=torch.float64, device=self.dev)
        self.h = torch.diag(self.onsite)
        self.S = torch.eye(self.n, dtype=torch.float64, device=self.dev)
        ij = (self.atom[:, None], self.atom[None, :], self.comp[:, None], self.comp[None, :])
        for T in itertools.product(range(-k, k + 1), repeat=3):
            own = eye if T == (0, 0, 0) else torch.zeros_like(eye)
            d = d0 + self.box * torch.tensor(T, dtype=torch.float64, device=self.dev)
            d = d + own[..., None]  # the atom itself: any length, masked below
            r = torch.sqrt((d * d).sum(-1))
            on = 1.0 - own
            x = torch.clamp(r / p["gamma_cut"], max=1.0)
            a = p["coulomb_k"] / p["hubbard_u"]
            self.G = self.G + on * p["coulomb_k"] / torch.sqrt(r * r + a * a) * (1 - x) ** 4 * (1 + 4 * x)
            self.E_pair = self.E_pair + 0.5 * (on * phi(r)).sum()
            l = d / r[..., None]
            self.h = self.h + blocks(on * hop(r), l)[ij]
            if p["overlap_s0"]:
                self.S = self.S - blocks(on * ovl(r), l)[ij]
        return self

    def H(self, n):
        v = (self.G @ n)[self.atom]
        return self.h + 0.5 * self.S * (v[:, None] + v[None, :])

    def diagonalise(self, H):
        if not self.p["overlap_s0"]:
            return torch.linalg.eigh(H)
        s, U = torch.linalg.eigh(self.S)
        Z = (U / torch.sqrt(s)) @ U.T
        e, C = torch.linalg.eigh(Z @ H @ Z)
        return e, Z @ C

    def charges(self, D):
        pop = (D * self.S).sum(1)
        return 2 * torch.zeros(self.N, dtype=torch.float64, device=self.dev).index_add_(0, self.atom, pop) - self.n0


def projector(e, C, occ):
    C = C[:, :int(round(occ))]
    return C @ C.T


def fermi(e, C, occ, kT):
    lo, hi = float(e[0]) - 40 * kT, float(e[-1]) + 40 * kT
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        lo, hi = (mu, hi) if float(torch.sigmoid((mu - e) / kT).sum()) < occ else (lo, mu)
    mu = 0.5 * (lo + hi)
    return (C * torch.sigmoid((mu - e) / kT)) @ C.T, mu


MOST = 4200  # orbitals that are diagonalised in a few seconds


def exact(case, seed):
    k = case["kind"]
    if k == "serve" or (k != "batch" and orbitals(case) > MOST):
        return None
    if k == "batch":
        out = []
        for i, N in enumerate(batch_sizes(case)):
            X = Exact(*liquid(int(N), 1000 * seed + i), PLAIN)
            out.append(projector(*torch.linalg.eigh(X.h), X.n_occ).reshape(-1))
        return torch.cat(out)
    if k in ("sp2", "bsr_sp2"):
        X = Exact(*liquid(case["atoms"], seed, morton=k == "bsr_sp2"), PLAIN)
        D = projector(*torch.linalg.eigh(X.h), X.n_occ)
        return D if k == "sp2" else {"D_rows": None, "D_cols": None, "D": None, "q": X.charges(D)}
    if k in ("fermi", "bsr_fermi"):
        R, types, box = vapour(case["molecules"], seed, morton=k == "bsr_fermi")
        X = Exact(R, types, box, PLAIN if k == "fermi" else GAPPED)
        H = X.H(torch.as_tensor(charges(types, seed, Q_PLAIN if k == "fermi" else Q_GAPPED), device=X.dev))
        D, mu = fermi(*torch.linalg.eigh(H), X.n_occ, case["kT"])
        if k == "fermi":
            # in a gap the trace holds for a range of mu: D is the result
            return {"D": D, "mu": None}
        return {"D_rows": None, "D_cols": None, "D": None, "q": X.charges(D), "mu": None}
    return exact_step(case, seed)


def exact_step(case, seed, device=None):
    k = case["kind"]
    p = OVERLAP if k == "nonorth" else GAPPED
    R, types, box = vapour(case["molecules"], seed, morton=k == "bsr_md")
    X = Exact(R, types, box, p, device)
    R, v, F, q, hist, m = (torch.as_tensor(a, dtype=torch.float64, device=X.dev)
                           for a in (R, *checkpoint(types, seed, Q_OVERLAP if k == "nonorth" else Q_GAPPED), masses(types)))
    v = v + 0.5 * DT * ACC * F / m[:, None]
    R = (R + DT * v).requires_grad_()
    n = 2 * hist[0] - hist[1] + KAPPA * (q - hist[0]) + ALPHA * sum(c * hist[j] for j, c in enumerate(CK))
    X.build(R)
    with torch.no_grad():
        H, S = X.H(n), X.S.detach()
        D = projector(*X.diagonalise(H), X.n_occ)
        W = D @ H @ D
        q = X.charges(D)
        V = (X.G @ n)[X.atom]
        A = V[:, None] * D + D * V[None, :] - 2 * W
    band, scc = 2 * (D * X.h).sum(), 0.5 * (2 * q - n) @ (X.G @ n)
    E = band + scc + X.E_pair
    on = E if not p["overlap_s0"] else E + (A * X.S).sum()
    F = -torch.autograd.grad(on, R)[0]
    v = v + 0.5 * DT * ACC * F / m[:, None]
    KE = 0.5 * (m[:, None] * v * v).sum() / ACC
    E, band, scc, pair = (float(x.detach()) for x in (E, band, scc, X.E_pair))
    en = torch.tensor([float(KE) + E, E, band, scc, pair, float(KE), float((n - q).abs().max()), 1.0],
                      dtype=torch.float64, device=X.dev)
    out = {"R": R.detach(), "v": v, "F": F, "q": q, "n": torch.cat([n[None], hist[:-1]]), "E": en}
    if k == "bsr_md":
        return dict(out, D_rows=None, D_cols=None, D=None)
    return dict(out, D=D) if k == "md" else dict(out, D=D, W=W, S=S)
