"""The workloads on which the library's speed is measured.

Each case is work that a user has the library do, through the calls of
paper_1402_7285_gb300: the block-sparse product, the panel solver (G, then
LDOS and density matrix), the local-subspace solver and the learned schedule.
Systems are the synthetic tight-binding models of `workloads`, with the seed of
the case; arrays are in device memory, as a program that keeps its matrices on
the GPU has them.

Solutions are compared at the solver's default tolerance, 1e-10, so that two
runs whose sums are ordered differently still agree; the energy broadening eta
then sets the number of iterations.  The iteration counts and the residuals at
the stopping step are not returned: they tell when a column stopped, and move
by some per cent with the last bit of any sum (the Krylov process has lost
orthogonality by then), while the Green's function does not.
"""
import math

import numpy as np
import torch

import paper_1402_7285_gb300 as tb
import workloads as wl
from paper_1402_7285_gb300 import scheduler

DEV = "cuda:0"
PREC = {"fp64": tb.TB_PREC_FP64, "mixed": tb.TB_PREC_MIXED, "df64": tb.TB_PREC_DF64}
BASE = {"anderson": wl.C1_SYSTEM, "sp3": wl.C2_SYSTEM, "fcc9": wl.C3_SYSTEM, "fcc4": wl.C4_SYSTEM,
        "subst": wl.C5_SYSTEM}
GRID = {"anderson": (-7.0, 7.0), "sp3": (-10.0, 6.0), "fcc9": (-8.0, 8.0), "fcc4": (-8.0, 8.0),
        "subst": (-10.0, 6.0)}


def listed():
    return [
        # a first look at a small scalar system: three vectors times a 1331-row matrix
        {"name": "spmm_f64_small", "kind": "spmm", "system": "anderson", "size": 11, "ncols": 3, "prec": "fp64"},
        # the product of the benchmark: sp3 matrix of 131072 rows, a full panel, FP32
        {"name": "spmm_f32_sp3", "kind": "spmm", "system": "sp3", "size": 32, "ncols": 64, "prec": "mixed"},
        # s+p+d orbitals on an open cluster, a panel width that fills half of the next compiled one
        {"name": "spmm_df64_fcc9", "kind": "spmm", "system": "fcc9", "size": 20011, "ncols": 33, "prec": "df64"},
        # the smallest solve: two orbitals of a 64-atom cell with overlap, eight energies
        {"name": "solve_small", "kind": "solve", "system": "sp3", "size": 4, "ncols": 2, "nz": 8, "eta": 0.05,
         "prec": "fp64", "solver": "cocg", "full": False},
        # the Anderson-model configuration, its first panel of columns, plain FP64
        {"name": "solve_anderson_f64", "kind": "solve", "system": "anderson", "size": 16, "ncols": 32, "nz": 32,
         "eta": 0.01, "prec": "fp64", "solver": "cocg", "full": False},
        # overlap in plain FP64, more columns than the panel has slots
        {"name": "solve_overlap_f64", "kind": "solve", "system": "sp3", "size": 11, "ncols": 40, "nz": 24,
         "eta": 0.3, "prec": "fp64", "solver": "cocg", "full": False},
        # the benchmark's panel (sp3, 131072 rows, overlap, 64 shifts, 64 columns, df64) at a broadening that a
        # contour or a smooth density of states takes; an iteration costs the same at any broadening
        {"name": "solve_bench_df64", "kind": "solve", "system": "sp3", "size": 32, "ncols": 64, "nz": 64,
         "eta": 0.5, "prec": "df64", "solver": "cocg", "full": False},
        # whole solution vectors (every row kept) of a few orbitals
        {"name": "solve_full_df64", "kind": "solve", "system": "sp3", "size": 9, "ncols": 6, "nz": 33, "eta": 0.3,
         "prec": "df64", "solver": "cocg", "full": True},
        # the second solver (QMR) on s+p+d blocks without overlap
        {"name": "solve_qmr_fcc9", "kind": "solve", "system": "fcc9", "size": 400, "ncols": 16, "nz": 48,
         "eta": 0.1, "prec": "fp64", "solver": "qmr", "full": False},
        # order-N work: truncated problems of uneven size on a cluster with vacancies and a surface, with overlap
        {"name": "local_fcc4_df64", "kind": "local", "system": "fcc4", "size": 60000, "ncols": 608, "nz": 64,
         "eta": 0.05, "prec": "df64", "rmin": 2, "rmax": 4},
        # the same with nine orbitals, no overlap; the largest subspaces exceed shared memory
        {"name": "local_fcc9_df64", "kind": "local", "system": "fcc9", "size": 20000, "ncols": 152, "nz": 128,
         "eta": 0.1, "prec": "df64", "rmin": 2, "rmax": 5},
        # the learned schedule: descriptors of the columns, training on their iteration counts, prediction
        {"name": "learn_schedule", "kind": "learn", "system": "fcc4", "size": 60000, "ncols": 4096, "batch": 256,
         "epochs": 4, "rmin": 2, "rmax": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmm", "spmm", "solve", "solve", "bench", "local", "local", "learn"])
    if kind == "spmm":
        system = rng.choice(["anderson", "sp3", "fcc9", "fcc4"])
        lo, hi = {"anderson": (5, 50), "sp3": (4, 32), "fcc9": (50, 20000), "fcc4": (100, 100000)}[system]
        return {"kind": "spmm", "system": system, "size": _log(rng, lo, hi), "ncols": _log(rng, 1, 64),
                "prec": rng.choice(["fp64", "mixed", "df64"])}
    if kind == "solve":  # to convergence, on systems whose dense solution is at hand
        system = rng.choice(["anderson", "sp3", "sp3", "subst", "fcc9"])
        lo, hi = {"anderson": (5, 16), "sp3": (3, 9), "subst": (3, 9), "fcc9": (20, 300)}[system]
        full = rng.random() < 0.2
        return {"kind": "solve", "system": system, "size": _log(rng, lo, hi), "ncols": _log(rng, 1, 6 if full else 48),
                "nz": _log(rng, 2, 64), "eta": rng.choice([0.2, 0.3, 0.5]), "prec": rng.choice(["fp64", "df64", "df64"]),
                "solver": rng.choice(["cocg", "cocg", "qmr"]), "full": full}
    if kind == "bench":  # vectors larger than the caches
        return {"kind": "solve", "system": rng.choice(["sp3", "subst"]), "size": rng.randint(17, 32),
                "ncols": _log(rng, 8, 64), "nz": _log(rng, 16, 64), "eta": rng.choice([0.5, 1.0]), "prec": "df64",
                "solver": "cocg", "full": False}
    rmin = rng.randint(1, 3)
    rmax = rng.randint(rmin, 4)
    if kind == "local":
        system = rng.choice(["fcc4", "subst", "fcc9"])
        size = rng.randint(10, 40) if system == "subst" else _log(rng, 3000, 60000)
        return {"kind": "local", "system": system, "size": size, "ncols": _log(rng, 20, 400), "nz": _log(rng, 8, 128),
                "eta": rng.choice([0.1, 0.2, 0.3]), "prec": rng.choice(["fp64", "df64", "df64"]), "rmin": rmin,
                "rmax": rmax}
    return {"kind": "learn", "system": "fcc4", "size": _log(rng, 6000, 60000), "ncols": _log(rng, 300, 4096),
            "batch": rng.choice([64, 128, 256, 1000]), "epochs": rng.randint(1, 4), "rmin": rmin, "rmax": rmax}


# ------------------------------------------------------------------ inputs
def _spec(case):
    base = BASE[case["system"]]
    return wl.scaled(base, **({"L": case["size"]} if base.lattice == wl.SC_PERIODIC else {"n_sites": case["size"]}))


def _pattern_rows(H, j):
    """Rows coupled to row j: all orbitals of the atoms in its block row (what the Mulliken form needs)."""
    a = int(j) // H.bdim
    cols = H.col_idx[H.row_ptr[a]:H.row_ptr[a + 1]].astype(np.int64)
    return (cols[:, None] * H.bdim + np.arange(H.bdim)).ravel()


def _dev(x):
    return torch.as_tensor(x, device=DEV)


def _host_inputs(case, seed):
    """Matrices, shifts, columns and kept rows (or subspaces) of a case, on the host."""
    H, S, _ = tb.build_system(_spec(case), int(seed))
    d = {"H": H, "S": S}
    rng = np.random.default_rng(int(seed))
    if case["kind"] == "spmm":
        return d
    n = min(case["ncols"], H.n_brows)
    lo, hi = GRID[case["system"]]
    if case["kind"] == "solve":
        # which orbitals is the case's own choice: the number of rows kept, and with it the outputs' shape, is its too
        cols = np.random.default_rng(case["size"]).choice(H.n_rows, n, replace=False)
        d["rhs"] = np.sort(cols).astype(np.int64)
        kept = [np.arange(H.n_rows) if case["full"] else _pattern_rows(H, j) for j in d["rhs"]]
        d["optr"] = np.concatenate([[0], np.cumsum([len(k) for k in kept])]).astype(np.int64)
        d["orows"] = np.concatenate(kept).astype(np.int64)
    else:
        radii = tuple(range(case["rmin"], case["rmax"] + 1))
        d["rhs"], d["rad"] = wl.sample_local_rhs(H.n_brows, H.bdim, n, radii, int(seed))
        d["sptr"], d["satoms"] = tb.local_subspaces(H, d["rhs"], d["rad"])
        d["optr"] = np.arange(n + 1, dtype=np.int64)
        d["orows"] = d["rhs"].copy()
    if case["kind"] == "learn":
        # log iteration counts: they grow with the subspace, with a spread of their own
        y = np.log(np.diff(d["sptr"]).astype(np.float64)) + 0.2 * rng.standard_normal(n)
        d["y"] = ((y - y.mean()) / (y.std() or 1.0)).astype(np.float32)
        d["params"] = scheduler.init_params(int(seed) & 0xffff)
    else:
        d["z"] = wl.midpoint_shifts(case["nz"], lo, hi, case["eta"])
        d["w"] = np.full(case["nz"], (hi - lo) / case["nz"])
        d["mu"], d["kT"] = 0.25, 0.1
    return d


def _panel(case, H, seed):
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return torch.randn(H.n_rows, case["ncols"], dtype=torch.complex128, device=DEV, generator=g)


def prepare(case, seed):
    d = _host_inputs(case, seed)
    st = {"case": case, "ctx": tb.Context(), "H": d["H"].to(DEV), "S": d["S"].to(DEV) if d["S"] is not None else None}
    if case["kind"] == "spmm":
        st["X"] = _panel(case, d["H"], seed)
    for k in ("rhs", "optr", "orows", "rad", "sptr", "satoms", "z", "w"):
        if k in d:
            st[k] = _dev(d[k])
    for k in ("mu", "kT", "y", "params"):
        if k in d:
            st[k] = d[k]
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case, ctx = st["case"], st["ctx"]
    if case["kind"] == "spmm":
        return tb.bsr_spmm(ctx, st["H"], st["X"], PREC[case["prec"]])
    if case["kind"] == "learn":
        # as scheduler.train and scheduler.predict do it: normalised descriptors, a fit, predictions for the columns
        D = tb.descriptors(ctx, st["H"], st["S"], st["rhs"], st["rad"], st["sptr"], st["satoms"])
        sd = D.std(dim=0, unbiased=False)
        X = (D - D.mean(dim=0)) / torch.where(sd > 1e-3, sd, torch.ones_like(sd))
        params, hist = tb.mlp_train(ctx, X.cpu().numpy(), st["y"], epochs=case["epochs"], batch=case["batch"], lr=2e-3,
                                    params=st["params"])
        # the loss history is a mean of FP32 squares
        return {"descriptors": D, "params": params, "loss": hist.astype(np.float32),
                "predicted": tb.mlp_predict(ctx, params, X)}
    if case["kind"] == "solve":
        r = tb.solve(ctx, st["H"], st["S"], st["z"], st["rhs"], st["optr"], st["orows"], precision=PREC[case["prec"]],
                     solver=tb.TB_SOLVER_QMR if case["solver"] == "qmr" else tb.TB_SOLVER_COCG)
        S = st["S"]
    else:
        r = tb.solve_local(ctx, st["H"], st["S"], st["z"], st["rhs"], st["sptr"], st["satoms"], st["optr"],
                           st["orows"], precision=PREC[case["prec"]])
        S = None  # only the column's own row is kept: the plain local density of states
    ldos, dm = tb.reduce_ldos_dm(ctx, r.G, st["z"], st["w"], st["mu"], st["kT"], st["rhs"], st["optr"], st["orows"], S)
    return {"G": r.G, "status": r.status, "ldos": ldos, "dm": dm}


# ------------------------------------------------------------------ work
def work(case):
    base = _spec(case)
    b = base.bdim
    deg = 7 if base.lattice == wl.SC_PERIODIC else 13
    atoms = base.L ** 3 if base.lattice == wl.SC_PERIODIC else int(base.n_sites * (1 - base.vacancy_frac))
    rows = atoms * b
    mat = atoms * deg * (8 * b * b + 4) + 8 * (atoms + 1)
    n_mat = 2 if base.has_overlap else 1
    if case["kind"] == "spmm":
        return {"bytes": mat + 2 * 16 * rows * case["ncols"], "flops": 4 * atoms * deg * b * b * case["ncols"]}
    n = case["ncols"]
    if case["kind"] == "learn":
        sub = {1: 10, 2: 40, 3: 90, 4: 180, 5: 300}
        mean = sum(sub[r] for r in range(case["rmin"], case["rmax"] + 1)) / (case["rmax"] - case["rmin"] + 1)
        steps = case["epochs"] * n
        return {"bytes": mat * n_mat + 4 * n * (mean + 32 + 32), "flops": 6 * 6200 * steps + n * mean * 10 * b * b * 10}
    kept = (rows if case["full"] else deg * b) if case["kind"] == "solve" else 1
    out = 16 * n * kept * case["nz"] + 8 * n * (kept + case["nz"])
    if case["kind"] == "local":
        sub = {1: 10, 2: 40, 3: 90, 4: 180, 5: 300}
        mean = sum(sub[r] for r in range(case["rmin"], case["rmax"] + 1)) / (case["rmax"] - case["rmin"] + 1)
        iters = 4 * math.sqrt(mean) / case["eta"]
        # the rows of one column: one product with H (and one with S) per iteration
        return {"bytes": mat * n_mat + out, "flops": n * iters * mean * 11 * n_mat * 4 * b * b}
    iters = min(150 / case["eta"], 3 * rows)
    # one product with H (and one with S) per iteration for every column; for panels larger than the caches, the
    # residual and the direction are read and written once per iteration
    vec = 16 * rows * n
    stream = 4 * vec * iters if vec > (64 << 20) else 0
    return {"bytes": mat * n_mat + out + stream, "flops": iters * atoms * deg * 4 * b * b * n * n_mat}


# ------------------------------------------------------------------ 64-bit references
def _dense(A, atoms=None):
    """Dense FP64 matrix of a block-sparse one (of its principal submatrix over `atoms`)."""
    b = A.bdim
    atoms = np.arange(A.n_brows) if atoms is None else np.asarray(atoms)
    loc = np.full(A.n_brows, -1, np.int64)
    loc[atoms] = np.arange(len(atoms))
    cnt = (A.row_ptr[atoms + 1] - A.row_ptr[atoms]).astype(np.int64)
    br = np.repeat(np.arange(len(atoms)), cnt)
    start = np.cumsum(cnt) - cnt
    k = np.arange(cnt.sum()) - np.repeat(start, cnt) + np.repeat(A.row_ptr[atoms], cnt)
    bc = loc[A.col_idx[k]]
    ok = bc >= 0
    br, bc, k = br[ok], bc[ok], k[ok]
    out = np.zeros((len(atoms), len(atoms), b, b))
    out[br, bc] = A.val[k]
    return _dev(out).permute(0, 2, 1, 3).reshape(len(atoms) * b, len(atoms) * b)


def _eig(H, S):
    """Eigenvalues and S-orthonormal eigenvectors: G(z) = Y (z - lam)^-1 Y^T."""
    if S is None:
        return torch.linalg.eigh(H)
    L = torch.linalg.cholesky(S)
    A = torch.linalg.solve_triangular(L, H, upper=False)
    A = torch.linalg.solve_triangular(L, A.T.contiguous(), upper=False)
    lam, V = torch.linalg.eigh(0.5 * (A + A.T))
    return lam, torch.linalg.solve_triangular(L.T.contiguous(), V, upper=True)


def _fermi(e, mu, kT):
    return 1.0 / (1.0 + np.exp(np.clip((e - mu) / kT, -700, 700)))


def _reduced(G, d, S):
    """LDOS and density-matrix elements of the kept entries."""
    optr, n = d["optr"], len(d["rhs"])
    col = np.repeat(np.arange(n), np.diff(optr))
    if S is None:
        wt = (d["orows"] == d["rhs"][col]).astype(np.float64)
    else:
        b = S.bdim
        i, j = d["orows"], d["rhs"][col]
        key = np.repeat(np.arange(S.n_brows), np.diff(S.row_ptr)) * S.n_brows + S.col_idx
        want = (i // b) * S.n_brows + j // b
        k = np.minimum(np.searchsorted(key, want), len(key) - 1)
        wt = np.where(key[k] == want, S.val[k, i % b, j % b], 0.0)
    im = G.imag
    ldos = torch.zeros(n, G.shape[1], dtype=torch.float64, device=DEV)
    ldos.index_add_(0, _dev(col), im * _dev(wt)[:, None])
    occ = _dev(d["w"] * _fermi(d["z"].real, d["mu"], d["kT"]))
    return -ldos / math.pi, -(im @ occ) / math.pi


def _exact_spmm(case, seed, d):
    H, X = d["H"], _panel(case, d["H"], seed)
    b = H.bdim
    br = _dev(np.repeat(np.arange(H.n_brows), np.diff(H.row_ptr)))
    val, ci = _dev(H.val), _dev(H.col_idx.astype(np.int64))
    Xr = torch.view_as_real(X).reshape(H.n_brows, b, -1)
    Y = torch.zeros_like(Xr)
    for s in range(0, H.nnzb, 100000):
        Y.index_add_(0, br[s:s + 100000], torch.bmm(val[s:s + 100000], Xr[ci[s:s + 100000]]))
    return torch.view_as_complex(Y.reshape(H.n_rows, -1, 2).contiguous())


def _exact_solve(case, d):
    H, S = d["H"], d["S"]
    if H.n_rows > 5500:
        return None
    lam, Y = _eig(_dense(H), _dense(S) if S is not None else None)
    inv = 1.0 / (_dev(d["z"])[None, :] - lam[:, None])
    G = torch.cat([(Y[_dev(d["orows"][d["optr"][c]:d["optr"][c + 1]])] * Y[int(j)]).to(torch.complex128) @ inv
                   for c, j in enumerate(d["rhs"])])
    ldos, dm = _reduced(G, d, S)
    return {"G": G, "status": None, "ldos": ldos, "dm": dm}


def _exact_local(case, d):
    H, S = d["H"], d["S"]
    rows = np.diff(d["sptr"]) * float(H.bdim)
    if (rows ** 3).sum() + 2e8 * len(rows) > 2e11:
        return None
    z, G = _dev(d["z"]), []
    for c, j in enumerate(d["rhs"]):
        at = d["satoms"][d["sptr"][c]:d["sptr"][c + 1]]
        lam, Y = _eig(_dense(H, at), _dense(S, at) if S is not None else None)
        jl = int(np.searchsorted(at, j // H.bdim)) * H.bdim + int(j % H.bdim)
        G.append(((Y[jl] ** 2)[:, None] / (z[None, :] - lam[:, None])).sum(0))
    G = torch.stack(G)
    ldos, dm = _reduced(G, d, None)
    return {"G": G, "status": None, "ldos": ldos, "dm": dm}


def _exact_descriptors(d):
    """The 26 local-environment numbers of each column (and six zeros)."""
    H, S, b = d["H"], d["S"], d["H"].bdim
    out = np.zeros((len(d["rhs"]), 32))
    for c, j in enumerate(d["rhs"]):
        at = d["satoms"][d["sptr"][c]:d["sptr"][c + 1]].astype(np.int64)
        n, a0 = len(at), int(j // b)
        cnt = (H.row_ptr[at + 1] - H.row_ptr[at]).astype(np.int64)
        br = np.repeat(np.arange(n), cnt)
        k = np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt) + np.repeat(H.row_ptr[at], cnt)
        bc = np.searchsorted(at, H.col_idx[k])
        ok = (bc < n) & (at[np.minimum(bc, n - 1)] == H.col_idx[k])
        br, bc, k = br[ok], bc[ok], k[ok]
        V, la, jo = H.val[k], int(np.searchsorted(at, a0)), int(j % b)
        dist = np.full(n, -1)
        dist[la] = 0
        for s in range(int(d["rad"][c])):
            new = bc[dist[br] == s]
            dist[new[dist[new] < 0]] = s + 1
        diag = V[br == bc][:, np.arange(b), np.arange(b)].ravel()
        hjj = diag[la * b + jo]
        mine = br == la
        srow = (S.val[k][mine][:, jo, :] ** 2).sum() - S.val[k][mine & (bc == la)][0, jo, jo] ** 2
        off = V[mine & (bc != la)]
        v, mom = np.zeros((n, b)), []
        v[la, jo] = 1.0
        for _ in range(5):
            y = np.zeros((n, b))
            np.add.at(y, br, np.einsum("kij,kj->ki", V, v[bc]))
            y -= hjj * v
            mom += [(v * v).sum(), (v * y).sum()]
            v = y
        o = out[c]
        o[0], o[1] = d["rad"][c] / 5.0, math.log(n) / math.log(1000.0)
        o[2:7] = [(dist == s).sum() / 100.0 for s in range(1, 6)]
        o[7], o[8] = (H.row_ptr[a0 + 1] - H.row_ptr[a0] - 1) / 12.0, hjj
        o[9:17] = [math.copysign(abs(mom[q]) ** (1.0 / q), mom[q]) for q in range(2, 10)]
        o[17:22] = srow, diag.mean(), diag.std(), diag.min(), diag.max()
        o[22] = (V[mine][:, jo, :] ** 2).sum() - hjj ** 2
        o[23] = np.sqrt((off ** 2).sum((1, 2))).mean() if len(off) else 0.0
        o[24], o[25] = n * b / 1000.0, (dist == dist.max()).mean()
    return out


def exact(case, seed):
    d = _host_inputs(case, seed)
    if case["kind"] == "spmm":
        return _exact_spmm(case, seed, d)
    if case["kind"] == "solve":
        return _exact_solve(case, d)
    if case["kind"] == "local":
        return _exact_local(case, d)
    # the fit sees FP16 forward weights and stops after a few epochs: no value of its own in 64 bits
    return {"descriptors": _dev(_exact_descriptors(d)), "params": None, "loss": None, "predicted": None}
