"""The work that users of this library have it do, as timed cases.

A case is one call sequence through the Python binding on inputs made on the GPU from a seed: a geometry step
(plan, chemical potential, density write-back), one bisection point on a plan that is kept, a step with forces, a
step on merged submatrices, the training of the bound predictor. Sizes, element model, options and basis are those
of the repository's workloads (synth/systems.py, synth/sites.py, bench.py and the GPU tests); the molecule counts
in between and the odd ones are generic.

Result types: the FP64 path's matrices come back as the library writes them (float64). The tensor-core modes'
matrices hold about six digits in a float64 buffer, and the program that asked for such a mode keeps them as
float32, which is what `run` returns.
"""
from types import SimpleNamespace

import numpy as np
import torch

import paper_2104_08245_gb300 as nl

DEV = "cuda"
SPACING, JITTER, CUTOFF = 3.1, 0.3, 6.0          # water's density on a cubic lattice, Angstrom
MOVE = 0.05                                      # displacement of a step within one neighbour list
S_EXP, HOP, HOP_LEN = 0.5, -0.2, 1.5             # S = exp(-S_EXP r^2), H0 = HOP exp(-r / HOP_LEN)
ONSITE_6 = (-1.0, -0.5, -0.5, -0.5, 0.3, 0.3)    # four occupied orbitals a molecule
OCC_6, OCC_23 = 4, 6
ONSITE_SITE = ((-1.0, -0.5, -0.5, -0.5), (-0.4, 0.3), (-1.2, 0.2, 0.2, 0.2))   # O, H, ion
OCC_SITE = (4, 1, 1)
MU_GAP = -0.1                                    # inside the gap of every system made here


def _water(name, n, precision, **kw):
    """A molecular system of n[0] x n[1] x n[2] molecules and how it is solved."""
    c = {"name": name, "kind": "step", "nx": n[0], "ny": n[1], "nz": n[2], "nbf": "6", "density": 0.0,
         "precision": precision, "inverse": "cholesky" if precision in ("fp64", "fp32") else "ns",
         "bound": "gershgorin"}
    c.update(kw)
    return c


def listed():
    return [
        # a single small cell solved to full precision, with the forces' matrix: the smallest call, and the
        # setting that every result is checked against
        _water("fp64_forces_64", (4, 4, 4), "fp64", kind="forces"),
        # a box of water of varying density to full precision: reference densities
        _water("fp64_step_1000", (10, 10, 10), "fp64", density=0.2),
        # one MD step of a small cell in the production mode: latency and launches
        _water("step_64", (4, 4, 4), "bf16x3"),
        # MD steps of ordinary boxes, submatrices of uneven size (114 to 294 rows)
        _water("step_4096_uneven", (16, 16, 16), "bf16x3", density=0.2),
        _water("step_32768_uneven", (32, 32, 32), "bf16x3", density=0.2),
        # the large production step (the benchmark's size)
        _water("step_262144", (64, 64, 64), "bf16x3"),
        # a step with forces in the tightest tensor-core mode, the elements generated on the device, ragged sizes
        _water("fp32_forces_2717", (13, 11, 19), "fp32", kind="forces", generate=True),
        # one chemical potential on a plan that is kept (a bisection driven by the caller, several ranks)
        _water("fp16_point_4096", (16, 16, 16), "fp16", kind="point"),
        # a larger basis: 23 functions a molecule, about 600 to 710 rows
        _water("step_512_split_valence", (8, 8, 8), "bf16x3", nbf="23"),
        # 6 or 23 functions a molecule, power-iteration bounds, a bracket that needs several points
        _water("mixed_343_power", (7, 7, 7), "bf16x3", nbf="mixed", bound="power", lo=-2.2, hi=1.3),
        # ions in water by atom, submatrices merged by the combination heuristic
        {"name": "grouped_sites_512", "kind": "grouped", "nx": 8, "ny": 8, "nz": 8, "ions": 0.02,
         "precision": "bf16x3", "inverse": "ns", "bound": "gershgorin"},
        # the learned bound predictor trained on the samples of a system
        {"name": "train_32768", "kind": "train", "samples": 32768, "batch": 1024, "epochs": 4},
    ]


def draw(rng):
    """One case of the same ranges: 27 to 100,000 molecules (the FP64 path to 1,000, the larger basis to 600)."""
    pick = rng.random()
    if pick < 0.1:
        return {"kind": "train", "samples": int(2 ** rng.uniform(11, 16)), "batch": rng.choice([256, 500, 1024, 4096]),
                "epochs": rng.randint(1, 4)}
    if pick < 0.2:
        return {"kind": "grouped", "nx": rng.randint(5, 9), "ny": rng.randint(5, 9), "nz": rng.randint(5, 9),
                "ions": round(rng.uniform(0.01, 0.05), 3), "precision": rng.choice(["bf16x3", "fp16"]), "inverse": "ns",
                "bound": "gershgorin"}

    def sides(lo, hi):
        edge = (2 ** rng.uniform(np.log2(lo), np.log2(hi))) ** (1 / 3)
        return tuple(max(3, round(edge * rng.uniform(0.8, 1.25))) for _ in range(3))
    kind = rng.choice(["step", "step", "forces", "point"])
    if pick < 0.4:
        c = _water("", sides(27, 800), "fp64", kind=kind, density=rng.choice([0.0, 0.2]))
    elif pick < 0.6:
        c = _water("", sides(27, 450), rng.choice(["bf16x3", "fp16", "fp32"]), kind=kind, nbf=rng.choice(["23", "mixed"]))
    else:
        density = rng.choice([0.0, 0.2])
        c = _water("", sides(27, 30000 if density else 100000), rng.choice(["bf16x3", "bf16x3", "fp16", "fp32"]),
                   kind=kind, density=density)
        if c["precision"] != "fp32":
            c["inverse"] = rng.choice(["ns", "ns", "cholesky"])
        if c["nx"] * c["ny"] * c["nz"] < 5000 and kind != "point" and rng.random() < 0.4:
            c["generate"] = True
    if kind != "point":
        c["bound"] = rng.choice(["gershgorin", "gershgorin", "power"])
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs

def _lattice(c, g):
    """Jittered lattice positions, with the local length scale varying by +- density where it is set."""
    dims = (c["nx"], c["ny"], c["nz"])
    f = dict(dtype=torch.float64, device=DEV)
    ijk = torch.stack(torch.meshgrid(*[torch.arange(d, device=DEV) for d in dims], indexing="ij"), -1)
    pos = ijk.to(torch.float64) * SPACING
    amp = c.get("density", 0.0)
    if amp:
        cd = [-(-d // 4) for d in dims]
        coarse = 1.0 + amp * (2.0 * torch.rand(cd, generator=g, **f) - 1.0)
        at = [ijk[..., k] * cd[k] / dims[k] for k in range(3)]
        i0 = [a.floor().long() for a in at]
        t = [a - b for a, b in zip(at, i0)]
        w = 0.0
        for corner in range(8):
            bit = [(corner >> k) & 1 for k in range(3)]
            wt = 1.0
            for k in range(3):
                wt = wt * (t[k] if bit[k] else 1.0 - t[k])
            w = w + wt * coarse[tuple((i0[k] + bit[k]) % cd[k] for k in range(3))]
        axes = []
        for k in range(3):
            gap = 0.5 * (w + w.roll(-1, k))
            axes.append((gap.cumsum(k) - gap) / gap.sum(k, keepdim=True) * dims[k] * SPACING)
        pos = torch.stack(axes, -1)
    pos = pos.reshape(-1, 3)
    cell = torch.tensor(dims, **f) * SPACING
    return pos + JITTER * (2.0 * torch.rand(pos.shape, generator=g, **f) - 1.0), cell, dims


def _pairs(pos, cell, radius, dims=None):
    """All ordered pairs (I, J), I == J included, with a minimum-image distance below (radius_I + radius_J) / 2, sorted
    by (I, J). dims: the lattice of `pos` when its sites are near their lattice points."""
    n = pos.shape[0]
    out_i, out_j = [], []

    def keep(I, J):
        d = pos[J] - pos[I]
        d = d - cell * torch.round(d / cell)
        r2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2]
        lim = 0.5 * (radius[I] + radius[J])
        at = torch.nonzero(r2 < lim * lim, as_tuple=True)
        I, J = torch.broadcast_tensors(I, J)
        out_i.append(I[at])
        out_j.append(J[at])

    all_j = torch.arange(n, device=DEV)
    if dims is not None and min(dims) >= 5:   # neighbours are at most two lattice steps away
        x, y, z = all_j // (dims[1] * dims[2]), all_j // dims[2] % dims[1], all_j % dims[2]
        for a in range(-2, 3):
            for b in range(-2, 3):
                for c in range(-2, 3):
                    keep(all_j, ((x + a) % dims[0] * dims[1] + (y + b) % dims[1]) * dims[2] + (z + c) % dims[2])
    else:
        for lo in range(0, n, 1024):
            keep(torch.arange(lo, min(n, lo + 1024), device=DEV)[:, None], all_j[None, :])
    I, J = torch.cat(out_i), torch.cat(out_j)
    order = torch.argsort(I * n + J)
    return I[order], J[order]


def _system(c, seed):
    """S and H0 block-CSR on the device (same pattern), positions, on-site energies and occupation. The box, its
    species and its neighbour list belong to the case; the seed moves every molecule by up to MOVE, one of the MD
    steps that share a neighbour list."""
    g = torch.Generator(device=DEV)
    g.manual_seed((c["nx"] * 1009 + c["ny"]) * 1013 + c["nz"])
    pos, cell, dims = _lattice(c, g)
    f = dict(dtype=torch.float64, device=DEV)
    n = pos.shape[0]
    if c["kind"] == "grouped":                 # by atom: O and two H, or an ion, on every lattice site
        ion = torch.rand(n, generator=g, **f) < c["ions"]
        q = torch.linalg.qr(torch.randn(n, 3, 3, generator=g, **f))[0]
        half = np.deg2rad(104.5) / 2
        h = [0.96 * (np.cos(half) * q[:, :, 0] + s * np.sin(half) * q[:, :, 1]) for s in (1, -1)]
        pos = torch.stack([pos, pos + h[0], pos + h[1]], 1).reshape(-1, 3)
        species = torch.stack([torch.where(ion, 2, 0), torch.ones_like(ion, dtype=torch.long), torch.ones_like(ion, dtype=torch.long)], 1)
        there = torch.stack([torch.ones_like(ion), ~ion, ~ion], 1).reshape(-1)
        pos, species = pos[there], species.reshape(-1)[there]
        n = pos.shape[0]
        table, occs, dims = [torch.tensor(o, **f) for o in ONSITE_SITE], OCC_SITE, None
        radius = torch.where(species == 2, 10.0, 6.0).to(torch.float64)
    else:
        low = torch.rand(OCC_23, generator=g, **f) * 0.4 - 1.0          # occupied levels, then empty ones
        high = torch.rand(23 - OCC_23, generator=g, **f) * 0.7 + 0.3
        table, occs = [torch.tensor(ONSITE_6, **f), torch.cat([low, high])], (OCC_6, OCC_23)
        big = torch.rand(n, generator=g, device=DEV) < 0.5
        species = {"6": torch.zeros_like(big), "23": torch.ones_like(big), "mixed": big}[c["nbf"]].long()
        radius = torch.full((n,), CUTOFF, **f)
        if c["density"]:
            dims = None
    nbf = torch.tensor([len(t) for t in table], device=DEV)[species]
    I, J = _pairs(pos, cell, radius, dims)
    g.manual_seed(int(seed))
    pos = torch.remainder(pos + MOVE * (2.0 * torch.rand(pos.shape, generator=g, **f) - 1.0), cell)
    d = pos[J] - pos[I]
    r = (d - cell * torch.round(d / cell)).square().sum(1).sqrt()
    size = nbf[I] * nbf[J]
    scale = 1.0 / torch.sqrt(size.to(torch.float64))
    row_ptr = torch.zeros(n + 1, dtype=torch.long, device=DEV)
    row_ptr[1:] = torch.bincount(I, minlength=n).cumsum(0)
    off = torch.zeros(I.shape[0] + 1, dtype=torch.long, device=DEV)
    off[1:] = size.cumsum(0)
    same = I == J
    s = torch.repeat_interleave(torch.where(same, 0.0, scale * torch.exp(-S_EXP * r * r)), size)
    h = torch.repeat_interleave(torch.where(same, 0.0, scale * HOP * torch.exp(-r / HOP_LEN)), size)
    first = torch.cumsum(nbf, 0) - nbf
    mol = torch.repeat_interleave(torch.arange(n, device=DEV), nbf)
    k = torch.arange(mol.shape[0], device=DEV) - first[mol]
    pad = torch.zeros(len(table), max(len(t) for t in table), **f)
    for a, t in enumerate(table):
        pad[a, :len(t)] = t
    onsite = pad[species[mol], k]
    diag = off[:-1][same][mol] + k * (nbf[mol] + 1)
    s[diag] = 1.0
    h[diag] = onsite
    i32 = lambda t: t.to(torch.int32).contiguous()  # noqa: E731
    return SimpleNamespace(
        nbf=i32(nbf), S=SimpleNamespace(row_ptr=i32(row_ptr), col_idx=i32(J), vals=s),
        H=SimpleNamespace(row_ptr=i32(row_ptr), col_idx=i32(J), vals=h), n_occ=float(torch.tensor(occs, device=DEV)[species].sum()),
        pos=pos, cell=cell, onsite=onsite, pairs=(I, J, off, first, mol), nvals=int(off[-1]))


def _options(c):
    return nl.options(c["precision"], inverse=1 if c["inverse"] == "ns" else 0,
                      bound_source=nl.BOUND_POWER if c["bound"] == "power" else nl.BOUND_GERSHGORIN)


def _groups(c, sysm):
    """The combination heuristic's groups, those wider than 64 functions cut in member order."""
    I, J = sysm.pairs[:2]
    nbf = sysm.nbf.cpu().numpy()
    g = nl.nolsm_combine_submatrices(sysm.nbf, sysm.S.row_ptr, sysm.S.col_idx).group_of.copy()
    order = np.argsort(g, kind="stable")
    start = width = -1
    label = -1
    for m in order:
        if g[m] != label or width + nbf[m] > 64:
            label, start, width = g[m], m, 0
        g[m], width = start, width + int(nbf[m])
    return g


def prepare(case, seed):
    if case["kind"] == "train":
        # features and targets as the method gives them on water: size, Gershgorin interval, neighbours, on-site
        # moments, chemical potential -> eigenvalue interval, steps / 16
        g = torch.Generator(device=DEV)
        g.manual_seed(int(seed))
        u = torch.rand(case["samples"], 7, generator=g, device=DEV)
        at = torch.tensor([1.1, -1.7, 0.6, 0.6, -0.37, 0.45, -0.15], device=DEV)
        by = torch.tensor([1.9, 0.4, 0.5, 0.8, 0.1, 0.1, 0.1], device=DEV)
        x = at + by * u
        t = torch.stack([0.8 * x[:, 1] - 0.1 * u[:, 3], 0.75 * x[:, 2] + 0.05 * u[:, 0], 0.55 + 0.1 * u[:, 1]], 1)
        mlp = nl.Mlp(int(seed) % 1000)
        return SimpleNamespace(case=case, mlp=mlp, x=x, t=t, start=mlp.get_params())
    sysm = _system(case, seed)
    st = SimpleNamespace(case=case, opts=_options(case), n_occ=sysm.n_occ)
    st.dsys = nl.DeviceSystem(sysm, DEV, values=not case.get("generate"))
    st.D = torch.zeros(sysm.nvals, dtype=torch.float64, device=DEV)
    if case["kind"] == "forces":
        st.W = torch.zeros_like(st.D)
    if case.get("generate"):
        st.model = nl.ElementModel(SimpleNamespace(
            pos=sysm.pos.cpu().numpy(), onsite=[sysm.onsite.cpu().numpy()], cell=sysm.cell.tolist(), dirs=None,
            spec=SimpleNamespace(s_exp=S_EXP, hop=HOP, hop_len=HOP_LEN, aniso=0.0)), DEV)
    if case["kind"] == "grouped":
        st.groups = _groups(case, sysm)
    if case["kind"] == "point":                # the plan and its geometry caches, as the bracket's call leaves them
        st.plan = nl.nolsm_build_submatrices(st.dsys)
        nl.nolsm_spectral_bracket(st.plan, st.opts)
    return st


def run(st):
    c = st.case
    if c["kind"] == "train":                   # from the same start each time: the trained weights and the losses
        st.mlp.set_params(st.start)
        losses = st.mlp.train(st.x, st.t, c["epochs"], c["batch"], 1e-3)
        return {"params": st.mlp.get_params(), "losses": np.asarray(losses, dtype=np.float32)}
    kept = (lambda m: m) if c["precision"] == "fp64" else (lambda m: m.float())
    if c["kind"] == "point":
        r = nl.nolsm_solve_batch(st.plan, MU_GAP, st.opts, check=True)
        st.plan.scatter(st.D)
        return {"D": kept(st.D), "trace_DS": r.trace_DS, "trace_DH": r.trace_DH, "t_S": kept(r.sub_t_S),
                "t_H": kept(r.sub_t_H), "status": r.sub_status}
    plan = nl.nolsm_build_submatrices(st.dsys)
    if c.get("generate"):
        nl.nolsm_plan_set_elements(plan, st.model)
    if c["kind"] == "grouped":
        grouped = nl.nolsm_build_grouped(plan, st.groups)
        r = nl.nolsm_solve_batch(grouped, MU_GAP, st.opts, per_sub=False, check=True)
        grouped.scatter(st.D)
        grouped.close()
        plan.close()
        return {"D": kept(st.D), "trace_DS": r.trace_DS, "trace_DH": r.trace_DH}
    r = plan.find_mu(st.n_occ, c.get("lo", 0.0), c.get("hi", 0.0), st.opts, check=True)
    plan.scatter(st.D)
    out = {"D": kept(st.D), "mu": r.mu, "trace_DS": r.trace_DS, "points": r.steps}
    if c["kind"] == "forces":
        plan.energy_weighted(st.W)
        out["W"] = kept(st.W)
    plan.close()
    return out


def work(case):
    """Method's count: 2 n^3 a product, two products a step, the overlap's inverse as five; inputs and results once."""
    if case["kind"] == "train":
        passes = case["epochs"] * case["samples"]
        return {"bytes": 40 * case["samples"] + 24 * 17923 * case["epochs"] * -(-case["samples"] // case["batch"]),
                "flops": 6 * 17923 * passes}
    n_mol = case["nx"] * case["ny"] * case["nz"]
    near = min(n_mol, 29.0)                    # molecules within the cutoff at water's density
    if case["kind"] == "grouped":
        sub, n, b, pairs = n_mol, 230.0, 8.0, 9 * n_mol * near
    else:
        b = {"6": 6.0, "23": 23.0, "mixed": 14.5}[case["nbf"]]
        sub, n, pairs = n_mol, near * b, n_mol * near
    values = pairs * (7.1 if case["kind"] == "grouped" else b * b)
    steps, products = (14, 0 if case["kind"] == "point" else 2) if case["precision"] == "fp64" else \
                      (10, 0 if case["kind"] == "point" else 5)
    out = values * (16 if case["kind"] == "forces" else 8)
    read = values * (0 if case.get("generate") else 16)
    if case["kind"] == "point":                # the prepared A_J in place of the elements
        read = sub * (n * n * (8 if case["precision"] == "fp64" else 4) + 3 * n * b * 8)
    return {"bytes": out + read, "flops": sub * (2 * steps + products) * 2.0 * n ** 3}


# ------------------------------------------------------------------------------------------------ in 64 bits

def exact(case, seed):
    """The densities in 64 bits with torch's batched products: every submatrix's sign by Newton-Schulz on dense
    gathered matrices (mu anywhere in the gap gives the same density)."""
    if case["kind"] == "train":
        return _exact_train(case, seed)
    sysm = _system(case, seed)
    I, J, off, first, mol = sysm.pairs
    nbf = sysm.nbf.long()
    n, nb = nbf.shape[0], mol.shape[0]
    if nb > (26000 if case.get("nbf", "6") == "6" else 12000):   # seconds, not minutes
        return None
    f = dict(dtype=torch.float64, device=DEV)
    # full dense S, H0 with one more row and column for the padding
    el = torch.arange(sysm.nvals, device=DEV)
    p = torch.repeat_interleave(torch.arange(I.shape[0], device=DEV), off[1:] - off[:-1])
    w = nbf[J[p]]
    a, b = (el - off[p]) // w, (el - off[p]) % w
    full = []
    for v in (sysm.S.vals, sysm.H.vals):
        m = torch.zeros(nb + 1, nb + 1, **f)
        m[first[I[p]] + a, first[J[p]] + b] = v
        full.append(m)
    if case["kind"] == "grouped":
        label = torch.as_tensor(_groups(case, sysm).astype(np.int64), device=DEV)
        _, group = torch.unique(label, return_inverse=True)
    else:
        group = torch.arange(n, device=DEV)
    ng = int(group.max()) + 1
    # rows of every group: the functions of all neighbours of its members, ascending
    near = torch.unique(group[J] * n + I)
    gi, mi = near // n, near % n
    fun_g = torch.repeat_interleave(gi, nbf[mi])
    loc = torch.arange(fun_g.shape[0], device=DEV)
    loc = loc - torch.repeat_interleave(torch.cumsum(nbf[mi], 0) - nbf[mi], nbf[mi])
    fun = first[torch.repeat_interleave(mi, nbf[mi])] + loc
    rows = torch.bincount(fun_g, minlength=ng)
    start = torch.cumsum(rows, 0) - rows
    D = torch.zeros(nb + 1, nb + 1, **f)
    W = torch.zeros(nb + 1, nb + 1, **f) if case["kind"] == "forces" else None
    t_S, t_H = torch.zeros(ng, **f), torch.zeros(ng, **f)
    order = torch.argsort(rows, descending=True)
    at = 0
    while at < ng:
        big = int(rows[order[at]])
        take = order[at:at + max(1, int(4e8 // (big * big)))]
        k = torch.arange(big, device=DEV)
        real = k[None, :] < rows[take][:, None]
        idx = torch.where(real, fun[(start[take][:, None] + k).clamp(max=fun.shape[0] - 1)], nb)
        eye = torch.eye(big, **f)
        S = full[0][idx[:, :, None], idx[:, None, :]] + eye * (~real)[:, None, :]
        H = full[1][idx[:, :, None], idx[:, None, :]] + eye * (~real)[:, None, :]
        Li = torch.linalg.solve_triangular(torch.linalg.cholesky(S), eye.expand_as(S), upper=False)
        Si = Li.transpose(1, 2) @ Li
        Si = Si @ (2.0 * eye - S @ Si)
        A = Si @ H
        X = A - MU_GAP * eye
        X = X / X.abs().sum(2).amax(1)[:, None, None]
        last = False
        for _ in range(80):
            V = eye - X @ X
            X = X + 0.5 * (X @ V)
            if last:
                break
            last = float(V.square().sum((1, 2)).max()) < 1e-12 * big
        P = 0.5 * (Si - X @ Si)
        mine = real & (group[mol][idx.clamp(max=nb - 1)] == take[:, None])
        t_S[take] = ((P * S).sum(1) * mine).sum(1)
        t_H[take] = ((P * H).sum(1) * mine).sum(1)
        g0, c0 = torch.nonzero(mine, as_tuple=True)
        D[idx[g0], idx[g0, c0][:, None].expand(-1, big)] = P[g0, :, c0]
        if W is not None:
            Wj = A @ P
            W[idx[g0], idx[g0, c0][:, None].expand(-1, big)] = Wj[g0, :, c0]
        at += take.shape[0]
    where = (first[I[p]] + a, first[J[p]] + b)
    out = {"D": D[where]}
    if W is not None:
        out["W"] = W[where]
    if case["kind"] in ("point", "grouped"):
        out["trace_DS"], out["trace_DH"] = float(t_S.sum()), float(t_H.sum())
    if case["kind"] == "point":
        out["t_S"], out["t_H"] = t_S, t_H
    return out


def _exact_train(case, seed):
    """The same minibatch Adam in 64 bits."""
    st = prepare(case, seed)
    x, t = st.x.double(), st.t.double()
    sizes = [(7, 128), (128,), (128, 128), (128,), (128, 3), (3,)]
    flat = torch.as_tensor(st.start, device=DEV).double()
    st.mlp.close()
    at, par = 0, []
    for s in sizes:
        k = int(np.prod(s))
        par.append(flat[at:at + k].reshape(s).clone().requires_grad_(True))
        at += k
    m, v = [torch.zeros_like(q) for q in par], [torch.zeros_like(q) for q in par]
    N, step, losses = case["samples"], 0, []
    for e in range(case["epochs"]):
        order = (torch.arange(N, device=DEV) * 7919 + e * 104729) % N
        total, count = 0.0, 0
        for lo in range(0, N, case["batch"]):
            xb, tb = x[order[lo:lo + case["batch"]]], t[order[lo:lo + case["batch"]]]
            y = torch.tanh(torch.tanh(xb @ par[0] + par[1]) @ par[2] + par[3]) @ par[4] + par[5]
            loss = (y - tb).square().sum() / (2 * xb.shape[0])
            grads = torch.autograd.grad(loss, par)
            step += 1
            with torch.no_grad():
                for q, gq, mq, vq in zip(par, grads, m, v):
                    mq.mul_(0.9).add_(gq, alpha=0.1)
                    vq.mul_(0.999).addcmul_(gq, gq, value=0.001)
                    q -= 1e-3 * (mq / (1 - 0.9 ** step)) / ((vq / (1 - 0.999 ** step)).sqrt() + 1e-8)
            total, count = total + loss.detach(), count + 1
        losses.append(float(total) / count)
    return {"params": torch.cat([q.detach().reshape(-1) for q in par]).cpu().numpy(),
            "losses": np.asarray(losses)}
