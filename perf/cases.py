"""The framework's measured cases: what its users have it do, through its public entry points.

Six kinds of work, over the range of sizes that the workloads, the tests and the benchmark of this
repository use:

* ``sigma``   -- the two-site effective Hamiltonian on a device vector (``apply_heff_device``), the
                 product that every local solver iterates, with the environments of the position in
                 place, as in a caller's own Lanczos or response solver;
* ``sigma1``  -- the one-site product on host arrays (``apply_heff1``);
* ``energy``  -- the FP64 energies of a loaded state (``load_mps`` of a checkpoint, ``energy``);
* ``window``  -- local updates of a sweep in both directions (``lcc_sweep_window``): right-hand side,
                 linear solve, truncation, environments, at the middle of the chain;
* ``program`` -- a whole calculation: DMRG reference, first-order sweeps, energies;
* ``gemm``    -- the allocation-free tensor-core product for callers that own all device memory.

A random state has sector dimensions spread around the mean electron number and spin as those of an
optimised state are (a few tens of sectors, the largest a sixth of the bond).  Every input comes from the
seed; the integrals of a workload are the repository's own.
"""
import functools
import math

import numpy as np
import torch

import paper_1509_00216_gb300 as mp
import synth

PRECS = {"fp64": mp.FP64, "tf32": mp.TF32, "bf16": mp.BF16, "bf16x3": mp.BF16X3, "bf16x6": mp.BF16X6}
OPS = {"H0_11": mp.OP_H0_11, "H_10": mp.OP_H_10, "U_11": mp.OP_U_11, "S_10": mp.OP_S_10, "H_11": mp.OP_H_11}


def listed():
    return [
        # The benchmark's workload and its inner product: the LCC matrix of the 24-orbital 3-band model at
        # the middle of the chain, split-BF16 operands; the largest product here.
        dict(name="sigma_threeband_bf16x3", kind="sigma", model="threeband", orbitals=24, M1=1500, M0=100, site=11,
             op="H0_11", prec="bf16x3", tc_env=False),
        # The same operator in the default precision of a context (FP64), at a middle size.
        dict(name="sigma_threeband_fp64", kind="sigma", model="threeband", orbitals=24, M1=500, M0=100, site=11,
             op="H0_11", prec="fp64", tc_env=False),
        # The transition product of a right-hand side (input in the reference's space), residual precision,
        # tensor-core environments, a position off the middle.
        dict(name="sigma_rhs_bf16x6", kind="sigma", model="threeband", orbitals=24, M1=450, M0=250, site=8,
             op="H_10", prec="bf16x6", tc_env=True),
        # The 2D lattice in TF32, the whole Hamiltonian's perturbation, an odd bond dimension.
        dict(name="sigma_hubbard2d_tf32", kind="sigma", model="hubbard2d", orbitals=16, M1=377, M0=64, site=7,
             op="U_11", prec="tf32", tc_env=False),
        # The smallest call: a short chain, where launches and host work are all there is.
        dict(name="sigma_chain_fp64", kind="sigma", model="chain", orbitals=8, M1=40, M0=16, site=3, op="H0_11",
             prec="fp64", tc_env=False),
        # One-site product on host arrays, as a caller on the CPU makes it.
        dict(name="sigma1_abinitio_fp64", kind="sigma1", model="abinitio", orbitals=14, M1=211, M0=50, site=7,
             op="H_11", prec="fp64", tc_env=False),
        # Energies of a checkpoint: FP64 passes over the whole chain.
        dict(name="energy_threeband", kind="energy", model="threeband", orbitals=24, M1=400, M0=150),
        dict(name="energy_abinitio", kind="energy", model="abinitio", orbitals=12, M1=150, M0=36),
        # Sweep steps at the middle of the chain, right and then left, on a determinant reference: mixed
        # precision (the benchmark's mode) and plain FP64.
        dict(name="window_abinitio_mixed", kind="window", model="abinitio", orbitals=16, M1=800, first=6, count=3,
             prec="bf16x3"),
        dict(name="window_abinitio_fp64", kind="window", model="abinitio", orbitals=16, M1=200, first=6, count=2,
             prec="fp64"),
        # A whole calculation on a short chain at exact bond dimension.
        dict(name="program_chain6_fp64", kind="program", orbitals=6, core=1, active=4, M0=16, M1=64, sweeps=2,
             prec="fp64"),
        # A ragged product without allocations.
        dict(name="gemm_noalloc_bf16x3", kind="gemm", m=1021, n=775, k=1502, prec="bf16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "sigma", "sigma1", "energy", "window", "program", "gemm"])
    if kind == "gemm":
        return dict(kind=kind, m=_log(rng, 17, 1021), n=_log(rng, 17, 775), k=_log(rng, 17, 1502),
                    prec=rng.choice(["bf16", "tf32", "bf16x3"]))
    if kind == "program":
        core = rng.choice([0, 1])
        return dict(kind=kind, orbitals=rng.choice([5, 6]), core=core, active=rng.choice([3, 4]), M0=16, M1=64,
                    sweeps=2, prec="fp64")
    model = rng.choice(["threeband", "hubbard2d", "abinitio", "chain"])
    k = {"threeband": 24, "hubbard2d": 16, "abinitio": rng.randrange(8, 15), "chain": rng.randrange(6, 17)}[model]
    top = {"threeband": 900, "hubbard2d": 377, "abinitio": 211, "chain": 377}[model]
    if kind == "window":
        k, prec = rng.choice([14, 16]), rng.choice(["bf16x3", "fp64"])
        return dict(kind=kind, model="abinitio", orbitals=k, M1=_log(rng, 40, 400 if prec == "bf16x3" else 200),
                    first=rng.randrange(k // 2 - 2, k // 2), count=rng.choice([1, 2]), prec=prec)
    if kind == "energy":
        return dict(kind=kind, model=model, orbitals=k, M1=_log(rng, 30, 150), M0=_log(rng, 8, 36))
    op = rng.choice(["H0_11", "H0_11", "H_10", "U_11", "S_10", "H_11"])
    prec = rng.choice(["fp64", "fp64", "bf16x3", "bf16x6", "tf32", "bf16"])
    M1 = _log(rng, 24, top if prec != "fp64" else min(top, 400))
    if kind == "sigma1":
        M1 = min(M1, 211)
    return dict(kind=kind, model=model, orbitals=k, M1=M1, M0=max(4, M1 // 5), site=rng.randrange(k // 4, 3 * k // 4), op=op,
                prec=prec, tc_env=rng.random() < 0.3)


# ---------------------------------------------------------------------------------------------------------
# inputs


@functools.lru_cache(maxsize=None)
def _model(model, k):
    """h, V, electrons, core and active orbitals of a workload."""
    if model == "threeband":
        c = synth.config(3)
    elif model == "hubbard2d":
        c = synth.config(2)
    elif model == "abinitio":
        h, V = synth.ab_initio(k, 3 * k, synth.SEED_BASE + 1)
        c = dict(n_orb=k, n_alpha=k // 2, n_beta=k // 2, n_core=k // 3, n_active=k // 3, h=h, V=V)
    else:
        h, V = synth.hubbard_chain(k, 1.0, 4.0)
        _, h, V = synth.to_orbital_basis(h, V)
        c = dict(n_orb=k, n_alpha=k // 2, n_beta=k // 2, n_core=k // 4, n_active=k // 2, h=h, V=V)
    return c


def _random_mps(k, n_elec, M, rng, masks, ncore, nact, centre=0):
    """A random block-sparse state in the format of ``load_mps``: bond sectors spread normally around the
    reference's mean electron number and spin, sites left of ``centre`` left-orthonormal, sites from it
    right-orthonormal."""
    left, right = synth._counts(masks), synth._counts(masks[::-1])
    bonds = []
    for b in range(k + 1):
        mean = 2 * min(b, ncore) + (n_elec - 2 * ncore) * min(max(b - ncore, 0), nact) / max(1, nact)
        secs = {}
        for q, cl in left[b].items():
            cr = right[k - b].get((n_elec - q[0], -q[1]), 0)
            if cr:
                secs[q] = (min(cl, cr), math.exp(-0.5 * ((q[0] - mean) / 1.1) ** 2 - 0.5 * (q[1] / 1.4) ** 2))
        norm = sum(w for _, w in secs.values())
        dims = {q: min(c, int(round(M * w / norm))) for q, (c, w) in secs.items()}
        if not any(dims.values()):
            dims = {max(secs, key=lambda q: secs[q][1]): 1}
        bonds.append([(q[0], q[1], d) for q, d in sorted(dims.items()) if d > 0])
    # sectors that no path through the chain reaches hold nothing
    keep = [{bonds[0][0][:2]}]
    for p in range(k):
        nxt = {(n + synth.LOCAL_N[s], z + synth.LOCAL_2SZ[s]) for (n, z) in keep[-1] for s in masks[p]}
        keep.append({q[:2] for q in bonds[p + 1]} & nxt)
    for p in range(k - 1, -1, -1):
        keep[p] &= {(n - synth.LOCAL_N[s], z - synth.LOCAL_2SZ[s]) for (n, z) in keep[p + 1] for s in masks[p]}
    bonds = [[q for q in b if q[:2] in kp] for b, kp in zip(bonds, keep)]
    sites = []
    for p in range(k):
        at = {q[:2]: j for j, q in enumerate(bonds[p + 1])}
        keys = [(ia, s, at[q]) for ia, (n, z, _) in enumerate(bonds[p]) for s in masks[p]
                if (q := (n + synth.LOCAL_N[s], z + synth.LOCAL_2SZ[s])) in at]
        side = 2 if p < centre else 0
        blocks = {}
        for g in sorted({key[side] for key in keys}):
            mine = [key for key in keys if key[side] == g]
            own = bonds[p + 1 if side else p][g][2]
            dims = [bonds[p if side else p + 1][key[2 - side]][2] for key in mine]
            X = rng.standard_normal((sum(dims), own))
            X = np.linalg.qr(X)[0] if sum(dims) >= own else X / math.sqrt(own)
            o = 0
            for key, d in zip(mine, dims):
                blocks[key] = np.ascontiguousarray(X[o:o + d] if side else X[o:o + d].T)
                o += d
        sites.append(blocks)
    return dict(bonds=bonds, sites=sites)


def _states(case, seed, centre=0):
    c = _model(case["model"], case["orbitals"])
    k, ne = c["n_orb"], c["n_alpha"] + c["n_beta"]
    rng = np.random.default_rng([seed, 7])
    ncore, nact = (ne // 2, 0) if case["kind"] == "window" else (c["n_core"], c["n_active"])
    phi1 = _random_mps(k, ne, case["M1"], rng, synth.site_masks(k), ncore, nact, centre)
    phi0 = _random_mps(k, ne, case.get("M0", 1), rng, synth.site_masks(k, ncore, nact, frozen=True), ncore, nact)
    return c, ncore, nact, phi0, phi1


def _context(c, ncore, nact, **kw):
    ctx = mp.Context(device=0, torch_memory=True, **kw)
    ctx.build_mpo(c["h"], c["V"], c["n_alpha"] + c["n_beta"], 0)
    ctx.set_spaces(ncore, nact)
    return ctx


def _chain(case, seed):
    """A Hubbard chain with on-site disorder, in its one-particle eigenbasis."""
    k = case["orbitals"]
    rng = np.random.default_rng([seed, 11])
    h, V = synth.hubbard_chain(k, 1.0, rng.uniform(1.5, 2.5))
    h = h + np.diag(rng.normal(0.0, 0.1, k))
    _, h, V = synth.to_orbital_basis(h, V)
    return dict(n_orb=k, n_alpha=case["core"] + case["active"] // 2, n_beta=case["core"] + case["active"] // 2, h=h, V=V)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        g = torch.Generator("cuda").manual_seed(seed)
        A = torch.randn(case["m"], case["k"], dtype=torch.float64, device="cuda", generator=g)
        B = torch.randn(case["n"], case["k"], dtype=torch.float64, device="cuda", generator=g)
        return dict(case=case, A=A, B=B, C=torch.empty(case["m"], case["n"], dtype=torch.float64, device="cuda"))
    if kind == "program":
        c = _chain(case, seed)
        ctx = mp.Context(device=0, prec=PRECS[case["prec"]], tol=1e-12)
        ctx.build_mpo(c["h"], c["V"], c["n_alpha"] + c["n_beta"], 0)
        ctx.set_spaces(case["core"], case["active"])
        return dict(case=case, ctx=ctx)
    if kind == "window":
        c, ncore, nact, phi0, phi1 = _states(case, seed, centre=case["first"])
        # one Hamiltonian of a scan over orbital energies
        shift = np.random.default_rng([seed, 3]).normal(0.0, 0.02, c["n_orb"])
        ctx = _context(dict(c, h=c["h"] + np.diag(shift)), ncore, nact, prec=PRECS[case["prec"]], tol=1e-8, max_iter=60)
        ctx.load_mps(0, phi0)
        ctx.dmrg_reference(1, 0)
        ctx.load_mps(1, phi1)
        return dict(case=case, ctx=ctx)
    c, ncore, nact, phi0, phi1 = _states(case, seed)
    ctx = _context(c, ncore, nact, tc_environments=case.get("tc_env", False))
    ctx.load_mps(0, phi0)
    if kind == "energy":
        ctx.dmrg_reference(case["M0"], 0)
        return dict(case=case, ctx=ctx, phi1=phi1)
    ctx.load_mps(1, phi1)
    site, op = case["site"], OPS[case["op"]]
    n_out, n_in = (ctx.local_dim1 if kind == "sigma1" else ctx.local_dim)(site, op)
    x = _vector(n_in, seed)
    if kind == "sigma1":
        ctx.apply_heff1(site, op, x, PRECS[case["prec"]])
        return dict(case=case, ctx=ctx, x=x)
    x, y = torch.from_numpy(x).cuda(), torch.empty(n_out, dtype=torch.float64, device="cuda")
    # one product: the environments of the position are in place, as they are for a solver's next product
    ctx.apply_heff_device(site, op, x.data_ptr(), y.data_ptr(), n_in, n_out, PRECS[case["prec"]])
    return dict(case=case, ctx=ctx, x=x, y=y)


def _vector(n, seed):
    x = np.random.default_rng([seed, 5]).standard_normal(n)
    return x / np.linalg.norm(x)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        A, B, C = state["A"], state["B"], state["C"]
        mp.tc_gemm_noalloc(0, torch.cuda.current_stream().cuda_stream, PRECS[case["prec"]], case["m"], case["n"],
                           case["k"], A.data_ptr(), B.data_ptr(), C.data_ptr())
        return C
    ctx = state["ctx"]
    if kind == "sigma":
        x, y = state["x"], state["y"]
        ctx.apply_heff_device(case["site"], OPS[case["op"]], x.data_ptr(), y.data_ptr(), x.numel(), y.numel(),
                              PRECS[case["prec"]])
        return y
    if kind == "sigma1":
        return ctx.apply_heff1(case["site"], OPS[case["op"]], state["x"], PRECS[case["prec"]])
    if kind == "energy":
        ctx.load_mps(1, state["phi1"])
        return _energies(ctx.energy())
    if kind == "window":
        first, n = case["first"], case["count"]
        right = ctx.lcc_window(case["M1"], first, n, 1)
        return dict(right=right, left=ctx.lcc_window(case["M1"], first + n - 1, n, -1))
    e0 = ctx.dmrg_reference(case["M0"], 3)
    j = ctx.lcc_sweep(case["M1"], case["sweeps"])
    return dict(_energies(ctx.energy()), reference=e0, sweep=j)


def _energies(e):
    return {key: e[key] for key in ("E0", "E2", "E3", "overlap01", "norm1")}


# ---------------------------------------------------------------------------------------------------------
# work that the paths cannot do without


@functools.lru_cache(maxsize=None)
def _tables(model, k, ncore, nact):
    """The operators' site tables (entries w0, w1, s_out, s_in and values) and channel charges per bond:
    input data of every contraction below, taken as given."""
    c = _model(model, k)
    with mp.Context(device=-1) as ctx:
        ctx.build_mpo(c["h"], c["V"], c["n_alpha"] + c["n_beta"], 0)
        ctx.set_spaces(ncore, nact)
        out = {}
        for name, which in (("H", mp.MPO_H), ("H0", mp.MPO_H0), ("U", mp.MPO_U), ("I", mp.MPO_ID)):
            sites = [ctx.export_mpo_site(which, p) for p in range(k)]
            charge = [{0: (0, 0)}]
            for idx, _ in sites:
                nxt = {}
                for w0, w1, so, si in np.unique(idx, axis=0):
                    q = charge[-1].get(int(w0))
                    if q is not None:
                        nxt[int(w1)] = (q[0] + synth.LOCAL_N[so] - synth.LOCAL_N[si],
                                        q[1] + synth.LOCAL_2SZ[so] - synth.LOCAL_2SZ[si])
                charge.append(nxt)
            out[name] = (sites, charge)
    return out


OPERATOR = {"H0_11": "H0", "H_10": "H", "U_11": "U", "S_10": "I", "H_11": "H"}


def _env_size(charge, bra, ket):
    """Values of an environment on one bond, and multiply-adds of one product of it with a ket-side matrix of
    the same sectors."""
    n = {}
    for q in charge.values():
        n[q] = n.get(q, 0) + 1
    size = mads = 0
    for (a, b, d) in bra:
        for (x, y, e) in ket:
            w = n.get((a - x, b - y), 0)
            size += w * d * e
            mads += w * d * e * e
    return size, mads


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=8 * (m * k + n * k + m * n), flops=2 * m * n * k)
    if kind == "program":
        # per sweep and position at least one product of the exact local problem and its environments
        k, M = case["orbitals"], case["M1"]
        pos = 2 * (k - 1) * (case["sweeps"] + 3)
        return dict(bytes=pos * 8 * 3 * M * M, flops=pos * 2 * 16 * M ** 3)
    c, ncore, nact, phi0, phi1 = _states(case, 0)
    k = c["n_orb"]
    tables = _tables(case["model"], k, ncore, nact)
    one = 2 if kind != "sigma1" else 1

    def product(name, bra, ket, l):
        charge = tables[name][1]
        (a, fa), (b, fb) = (_env_size(charge[i], bra["bonds"][i], ket["bonds"][i]) for i in (l, l + one))
        n = 4 ** one * 0.25 * sum(d for *_, d in ket["bonds"][l]) * sum(d for *_, d in ket["bonds"][l + one]) / 6
        return 8 * (a + b + 2 * n), 2 * 4 ** one * min(fa, fb)

    if kind in ("sigma", "sigma1"):
        ket = phi0 if case["op"].endswith("10") else phi1
        b, f = product(OPERATOR[case["op"]], phi1, ket, case["site"])
        return dict(bytes=b, flops=f)
    if kind == "window":
        f = b = 0
        for l in range(case["first"], case["first"] + case["count"]):
            x, y = product("H0", phi1, phi1, l)
            b, f = b + 2 * 2 * x, f + 2 * 3 * y   # both directions: two products and an environment update each
        return dict(bytes=b, flops=f)
    f = b = 0
    for name, bra, ket in (("H0", phi1, phi1), ("U", phi1, phi1), ("H", phi1, phi0), ("H0", phi1, phi0)):
        for i in range(1, k):
            s, mads = _env_size(tables[name][1][i], bra["bonds"][i], ket["bonds"][i])
            b, f = b + 8 * s, f + 2 * 2 * 4 * mads
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------------------------------------
# the same numbers in 64 bits by plain contraction


def _contract(table, bra, ket, k):
    """<bra|O|ket>, site by site over the operator's tables; differentiable in the tensors of ``bra``."""
    sites, charge = table
    env = {(0, 0): torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")}

    def classes(ch):
        out = {}
        for w in sorted(ch):
            out.setdefault(ch[w], {})[w] = len(out.get(ch[w], ()))
        return out

    for p in range(k):
        idx, val = sites[p]
        c0, c1 = classes(charge[p]), classes(charge[p + 1])
        mats = {}
        ent = {}
        for (w0, w1, so, si), v in zip(idx.tolist(), val.tolist()):
            q = charge[p].get(w0)
            if q is not None:
                ent.setdefault((q, so, si), []).append((w0, w1, v))
        for (q, so, si), es in ent.items():
            q1 = charge[p + 1][es[0][1]]
            m = np.zeros((len(c1[q1]), len(c0[q])))
            for w0, w1, v in es:
                m[c1[q1][w1], c0[q][w0]] += v
            mats[(q, so, si)] = torch.from_numpy(m).cuda()
        kb, bb = {}, {}
        for (ia, s, ib), t in ket["sites"][p].items():
            kb.setdefault(ia, []).append((s, ib, t))
        for (ia, s, ib), t in bra["sites"][p].items():
            bb.setdefault(ia, {})[s] = (ib, t)
        mid = {}
        for (ib, ik), L in env.items():
            qb, qk = bra["bonds"][p][ib], ket["bonds"][p][ik]
            q = (qb[0] - qk[0], qb[1] - qk[1])
            for si, jk, t in kb.get(ik, ()):
                X = None
                for so in bb.get(ib, ()):
                    m = mats.get((q, so, si))
                    if m is None:
                        continue
                    X = L @ t if X is None else X
                    Y = (m @ X.reshape(X.shape[0], -1)).reshape(m.shape[0], X.shape[1], X.shape[2])
                    key = (ib, so, jk)
                    mid[key] = mid[key] + Y if key in mid else Y
        env = {}
        for (ib, so, jk), Y in mid.items():
            jb, t = bb[ib][so]
            Z = t.T @ Y
            env[(jb, jk)] = env[(jb, jk)] + Z if (jb, jk) in env else Z
    return env[(0, 0)].sum() if env else torch.zeros((), dtype=torch.float64, device="cuda")


def _on_gpu(m):
    return dict(bonds=m["bonds"], sites=[{key: torch.from_numpy(t).cuda() for key, t in s.items()} for s in m["sites"]])


def _fused(m, l, local=None):
    """The state with bond l + 1 opened to the whole space of (bond l, site l), the two-site tensor being
    ``local`` (zeros without one), in the local layout: (state, the tensor's blocks in layout order)."""
    LN, LZ = synth.LOCAL_N, synth.LOCAL_2SZ
    mask = m["masks"]
    rows, cols = {}, {}
    for s in mask[l]:
        for ia, (n, z, d) in enumerate(m["bonds"][l]):
            rows.setdefault((n + LN[s], z + LZ[s]), []).append((ia, s, d))
    for s in mask[l + 1]:
        for ib, (n, z, d) in enumerate(m["bonds"][l + 2]):
            cols.setdefault((n - LN[s], z - LZ[s]), []).append((s, ib, d))
    qs = [q for q in sorted(rows) if q in cols]
    bond, first, second, order, at = [], {}, {}, [], 0
    for j, q in enumerate(qs):
        nr, nc = sum(r[2] for r in rows[q]), sum(x[2] for x in cols[q])
        bond.append((q[0], q[1], nr))
        eye, o = torch.eye(nr, dtype=torch.float64, device="cuda"), 0
        for ia, s, d in rows[q]:
            first[(ia, s, j)] = eye[o:o + d]
            o += d
        M = torch.zeros(nr, nc, dtype=torch.float64, device="cuda") if local is None else local[at:at + nr * nc].reshape(nr, nc)
        at += nr * nc
        M.requires_grad_(local is None)
        order.append(M)
        o = 0
        for s, ib, d in cols[q]:
            second[(j, s, ib)] = M[:, o:o + d]
            o += d
    bonds, sites = list(m["bonds"]), list(m["sites"])
    bonds[l + 1], sites[l], sites[l + 1] = bond, first, second
    return dict(bonds=bonds, sites=sites), order


def _opened1(m, l, local=None):
    """The state with the tensor of site l replaced by ``local`` (zeros without one), left-fused layout."""
    rows = {}
    for s in m["masks"][l]:
        for ia, (n, z, d) in enumerate(m["bonds"][l]):
            rows.setdefault((n + synth.LOCAL_N[s], z + synth.LOCAL_2SZ[s]), []).append((ia, s, d))
    site, order, at = {}, [], 0
    for ib, (n, z, d) in enumerate(m["bonds"][l + 1]):
        if (n, z) not in rows:
            continue
        nr = sum(r[2] for r in rows[(n, z)])
        M = torch.zeros(nr, d, dtype=torch.float64, device="cuda") if local is None else local[at:at + nr * d].reshape(nr, d)
        at += nr * d
        M.requires_grad_(local is None)
        order.append(M)
        o = 0
        for ia, s, e in rows[(n, z)]:
            site[(ia, s, ib)] = M[o:o + e]
            o += e
    sites = list(m["sites"])
    sites[l] = site
    return dict(bonds=m["bonds"], sites=sites), order


def _determinants(case, seed):
    """E0, E2, E3 of the chain in the space of all determinants (exact bond dimension)."""
    c = _chain(case, seed)
    k, na = c["n_orb"], c["n_alpha"]
    h, V = torch.from_numpy(c["h"]).cuda(), torch.from_numpy(np.ascontiguousarray(c["V"])).cuda()
    strings = [s for s in range(1 << k) if bin(s).count("1") == na]
    at = {s: i for i, s in enumerate(strings)}
    n = len(strings)
    A = np.zeros((k, k, n, n))
    for s in strings:
        for q in range(k):
            if s >> q & 1:
                for p in range(k):
                    t = s ^ (1 << q)
                    if not t >> p & 1:
                        sign = (-1) ** (bin(s & ((1 << q) - 1)).count("1") + bin(t & ((1 << p) - 1)).count("1"))
                        A[p, q, at[t | 1 << p], at[s]] += sign
    A = torch.from_numpy(A).cuda()
    T = h - 0.5 * torch.einsum("prrq->pq", V)
    G = torch.einsum("pqrs,rsab->pqab", V, A)
    one = torch.einsum("pq,pqab->ab", T, A) + 0.5 * torch.einsum("pqab,pqbc->ac", A, G)
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    H = torch.kron(one, eye) + torch.kron(eye, one) + torch.einsum("pqab,pqcd->acbd", A, G).reshape(n * n, n * n)
    lo, up = (1 << case["core"]) - 1, ~((1 << (case["core"] + case["active"])) - 1)
    cls = torch.tensor([(bin(a & lo).count("1") + bin(b & lo).count("1")) * 100 +
                        bin(a & up & ((1 << k) - 1)).count("1") + bin(b & up & ((1 << k) - 1)).count("1")
                        for a in strings for b in strings], device="cuda")
    H0 = H * (cls[:, None] == cls[None, :])
    ref = torch.nonzero(cls == 200 * case["core"]).flatten()
    w, v = torch.linalg.eigh(H0[ref][:, ref])
    phi0 = torch.zeros(n * n, dtype=torch.float64, device="cuda")
    phi0[ref] = v[:, 0]
    e0 = w[0]
    P = torch.outer(phi0, phi0)
    b = -(H @ phi0 - e0 * phi0)
    x = torch.linalg.solve(H0 - e0 * torch.eye(n * n, dtype=torch.float64, device="cuda") + P, b)
    x = x - phi0 * (phi0 @ x)
    e2, e3 = -(x @ b), x @ ((H - H0) @ x)
    return float(e0), float(e2), float(e3), float(x @ x)


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        s = prepare(case, seed)
        return s["A"] @ s["B"].T
    if kind == "window":
        return None   # the iterate of an inexact solve and a truncation: no 64-bit value of its own
    if kind == "program":
        e0, e2, e3, n1 = _determinants(case, seed)
        return dict(E0=e0, E2=e2, E3=e3, overlap01=None, norm1=n1, reference=e0, sweep=e2)
    c, ncore, nact, phi0, phi1 = _states(case, seed)
    k = c["n_orb"]
    if (kind == "energy" and k * case["M1"] > 10000) or case["M1"] > 600:
        return None   # over 20 seconds
    tables = _tables(case["model"], k, ncore, nact)
    for m, masks in ((phi0, [tuple(sorted({key[1] for key in s})) for s in phi0["sites"]]), (phi1, synth.site_masks(k))):
        m["masks"] = masks
    masks0, masks1 = phi0["masks"], phi1["masks"]
    phi0, phi1 = dict(_on_gpu(phi0), masks=masks0), dict(_on_gpu(phi1), masks=masks1)
    if kind == "energy":
        val = lambda name, a, b: float(_contract(tables[name], a, b, k))
        n00 = val("I", phi0, phi0)
        e0 = val("H0", phi0, phi0) / n00
        A, N1, s = val("H0", phi1, phi1), val("I", phi1, phi1), val("I", phi1, phi0)
        g, h = val("H", phi1, phi0), val("H0", phi1, phi0)
        e2 = A - e0 * N1 - 2 * s * (h - e0 * s) + 2 * (g - s * e0)
        return dict(E0=e0, E2=e2, E3=val("U", phi1, phi1) - 2 * s * (g - h), overlap01=s, norm1=N1)
    opened = _opened1 if kind == "sigma1" else _fused
    base = phi0 if case["op"].endswith("10") else phi1
    n_in = sum(M.numel() for M in opened(base, case["site"])[1])
    x = torch.from_numpy(_vector(n_in, seed)).cuda()
    with torch.no_grad():
        ket, _ = opened(base, case["site"], x)
    bra, blocks = opened(phi1, case["site"])
    value = _contract(tables[OPERATOR[case["op"]]], bra, ket, k)
    if not value.requires_grad:
        sigma = torch.zeros(sum(M.numel() for M in blocks), dtype=torch.float64, device="cuda")
    else:
        grads = torch.autograd.grad(value, blocks, allow_unused=True)
        sigma = torch.cat([(torch.zeros_like(M) if g is None else g).reshape(-1) for g, M in zip(grads, blocks)])
    return sigma.cpu().numpy() if kind == "sigma1" else sigma
