"""The work that a user of this framework has it do, as measurable cases.

Every case is one pass through the public entry points: a single operation on a bond (projected
Hamiltonian, its gradient, environment update, two-site split) or a call of the stateful engine.
Bonds and couplings are those of the repository's own models (`workloads`): Heisenberg chains, the
24x8 square and 12x6 triangular cylinders, the 16x8 J-Q2 cylinder, the transverse-field Ising chain
and the random-field cylinder of the region tests, at the bond dimensions that the benchmark and
the tests use and odd ones between them.

A split's singular vectors are unique only up to a sign, so a split case returns the wavefunction
that its factors make, A diag(lambda) B, sector matrix by sector matrix, beside lambda, the kept
dimensions and the kept weight.  The mixed-precision modes compute in FP32 (or on FP32
accumulators) and only hand their values over in FP64 buffers: those come back as float32.
"""
import functools
import math

import numpy as np
import torch

import paper_1301_3494_gb300 as pd
import workloads as wl

PRECS = {"fp64": pd.FP64, "tf32": pd.TF32, "bf16": pd.BF16}

# Charge widths (in 2 S^z) of a ground state's Schmidt spectrum, as the benchmark and tests take them.
SIGMA = {"chain": 3.0, "square": 5.0, "tri": 5.0, "jq2": 4.0, "tfim": None, "field": 4.0}


@functools.lru_cache(maxsize=None)
def _mpo(model):
    if model == "chain":
        return wl.heisenberg_chain(200)
    if model == "square":
        return wl.heisenberg_square_cylinder(24, 8)
    if model == "tri":
        return wl.heisenberg_triangular_cylinder(12, 6)
    if model == "jq2":
        return wl.jq2_cylinder(16, 8)[0]
    if model == "tfim":
        return wl.tfim_chain(128, 1.0, 0.7)
    return wl.field_square_cylinder(6, 4, seed=3)


@functools.lru_cache(maxsize=None)
def _bonds(model, m):
    mpo = _mpo(model)
    qn = list(mpo.site.qn)
    return wl.consistent_sectors(wl.bond_sectors(mpo.L, qn, mpo.qtot, m, SIGMA[model]), qn)


def _site_of(model, place):
    """Left site of a two-site window at `place` (0..1) of the lattice."""
    L = _mpo(model).L
    return min(L - 3, max(1, int(place * L)))


def listed():
    return [
        # a chain program's innermost call: tiny blocks, launch and call latency
        {"name": "heff_fp64_chain_m64", "kind": "heff", "model": "chain", "m": 64, "place": 0.5, "prec": "fp64"},
        # the exact (FP64) solves next to region boundaries and in merges
        {"name": "heff_fp64_square_m500", "kind": "heff", "model": "square", "m": 500, "place": 0.5, "prec": "fp64"},
        # the triangular cylinder in tf32, a bond dimension that is no multiple of anything
        {"name": "heff_tf32_tri_m1001", "kind": "heff", "model": "tri", "m": 1001, "place": 0.45, "prec": "tf32"},
        # the benchmark's bond and matvec
        {"name": "heff_bf16_square_m2000", "kind": "heff", "model": "square", "m": 2000, "place": 0.5, "prec": "bf16"},
        # forward and backward through the matvec for Hamiltonian learning (many MPO channels)
        {"name": "grad_jq2_m128", "kind": "grad", "model": "jq2", "m": 128, "place": 0.5},
        # growing a block by one site: FP64 on a chain, FP32 on the benchmark's bond
        {"name": "env_left_fp64_chain_m512", "kind": "env", "model": "chain", "m": 512, "place": 0.5,
         "side": "left", "prec": "fp64"},
        {"name": "env_right_bf16_square_m2000", "kind": "env", "model": "square", "m": 2000, "place": 0.5,
         "side": "right", "prec": "bf16"},
        # the split of a step: FP64, the merges' accurate split, and the benchmark's batch of the
        # four regions' mixed-precision splits
        {"name": "split_fp64_chain_m512", "kind": "split", "model": "chain", "m": 512, "bonds": 1, "mode": 0},
        {"name": "split_accurate_square_m1000", "kind": "split", "model": "square", "m": 1000, "bonds": 1, "mode": 1},
        {"name": "split_mixed4_square_m2000", "kind": "split", "model": "square", "m": 2000, "bonds": 4, "mode": 2},
        # whole programs: load a state and sweep a small chain in FP64; one parallel sweep of four
        # regions in the benchmark's mixed precision
        {"name": "sweep_fp64_chain_L16_m64", "kind": "sweep", "L": 16, "m": 64},
        {"name": "regions_bf16_field_m128", "kind": "regions", "m": 128, "regions": 4},
    ]


def draw(rng):
    kind = rng.choice(["heff", "heff", "env", "env", "split", "split", "grad", "sweep"])
    logu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    if kind in ("heff", "env"):
        prec = rng.choice(["fp64", "tf32", "bf16"])
        model = rng.choice(["chain", "square", "tri"])
        top = {"heff": 700, "env": 900}[kind] if prec == "fp64" else 1900
        c = {"kind": kind, "model": model, "m": logu(40, top), "place": round(rng.uniform(0.3, 0.7), 3), "prec": prec}
        if kind == "env":
            c["side"] = rng.choice(["left", "right"])
        return c
    if kind == "split":
        mode = rng.choice([0, 1, 2, 2])
        return {"kind": kind, "model": rng.choice(["chain", "square"]), "bonds": rng.choice([1, 2, 4]) if mode == 2 else 1,
                "m": logu(60, 1900 if mode == 2 else 700), "mode": mode}
    if kind == "grad":
        return {"kind": kind, "model": rng.choice(["chain", "tfim", "square"]), "m": logu(24, 160),
                "place": round(rng.uniform(0.3, 0.7), 3)}
    return {"kind": kind, "L": 2 * rng.randrange(5, 11), "m": logu(32, 64)}


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _env_keys(bond, flux):
    return [(q, w) for q in bond for w in range(len(flux)) if (q - int(flux[w])) in bond]


def _psi_keys(bl, br, qn):
    return [(q, s1, s2) for q in bl for s1 in range(len(qn)) for s2 in range(len(qn)) if q + qn[s1] + qn[s2] in br]


def _site_keys(bl, br, qn):
    return [(q, s) for q in bl for s in range(len(qn)) if q + qn[s] in br]


def _env_input(g, bond, flux, unit):
    """A projected-operator environment: the channel `unit` (nothing placed yet, or everything
    placed, on that side) is the identity, the other operators have entries of order one over the
    root of the block size."""
    parts = []
    for q, w in _env_keys(bond, flux):
        k = bond[q - int(flux[w])]
        if w == unit:
            parts.append(torch.eye(bond[q], k, dtype=torch.float64, device="cuda").reshape(-1))
        else:
            parts.append((_randn(g, bond[q], k) / math.sqrt(k)).reshape(-1))
    return torch.cat(parts)


def _psi_input(g, bl, br, qn):
    n = sum(bl[q] * br[q + qn[a] + qn[b]] for q, a, b in _psi_keys(bl, br, qn))
    x = _randn(g, n)
    return x / torch.linalg.vector_norm(x)


def _window(case):
    mpo = _mpo(case["model"])
    j = _site_of(case["model"], case["place"])
    bonds = _bonds(case["model"], case["m"])
    return mpo, list(mpo.site.qn), j, bonds[j], bonds[j + 1], bonds[j + 2]


def _isometry(g, rows, cols):
    return torch.linalg.qr(_randn(g, rows, cols))[0]


def _split_sites(case):
    L = _mpo(case["model"]).L
    n = case["bonds"]
    return [L // 2 - 1] if n == 1 else [L * (2 * i + 1) // (2 * n) - 1 for i in range(n)]


def _split_sectors(bl, br, qn):
    """Middle charge -> ([row blocks (q, s1)], [column blocks (s2, q_right)]), both ascending."""
    secs = {}
    for q, s1, s2 in _psi_keys(bl, br, qn):
        rows, cols = secs.setdefault(q + qn[s1], (set(), set()))
        rows.add((q, s1))
        cols.add((s2, q + qn[s1] + qn[s2]))
    return {qm: (sorted(r), sorted(c)) for qm, (r, c) in sorted(secs.items())}


def _split_input(g, bl, bm, br, qn, floor):
    """A two-site wavefunction as a local solve leaves it: the state kept so far (the middle
    bond's m values, decaying over three decades, outer charges lower) plus the new directions of
    the solve below it, down to 10^-floor."""
    blocks = {}
    qmax = max(1, max(abs(q) for q in bm))
    for qm, (rows, cols) in _split_sectors(bl, br, qn).items():
        r = sum(bl[q] for q, _ in rows)
        c = sum(br[q] for _, q in cols)
        n = min(r, c)
        k = min(n, bm.get(qm, 0))
        u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 0.8
        a = 1.5 * min(1.0, abs(qm) / qmax) ** 2
        i = torch.arange(n, device="cuda", dtype=torch.float64)
        s = torch.where(i < k, a + (3.0 - a) * (i + u) / max(k, 1), 3.5 + (floor - 3.5) * (i - k + u) / max(n - k, 1))
        M = (_isometry(g, r, n) * 10.0 ** -s) @ _isometry(g, c, n).T
        ro = 0
        for q, s1 in rows:
            co = 0
            for s2, qc in cols:
                blocks[(q, s1, s2)] = M[ro: ro + bl[q], co: co + br[qc]].reshape(-1)
                co += br[qc]
            ro += bl[q]
    psi = torch.cat([blocks[k] for k in _psi_keys(bl, br, qn)])
    return psi / torch.linalg.vector_norm(psi)


def _engine(mpo, precision, **more):
    W, flux, D = wl.pack_mpo(mpo)
    return pd.Engine(W, flux, D, list(mpo.site.qn), mpo.qtot, precision, 8, **more)


def _packed(mps, qn):
    return np.concatenate([wl.pack_site(mps.sites[j], mps.bonds[j], mps.bonds[j + 1], qn) for j in range(len(mps.sites))])


REGION_SWEEP = dict(dav_tol=1e-9, dav_max_iter=4, refine_iters=1, serial_regions=2)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        mpo = wl.heisenberg_chain(case["L"])
        qn = list(mpo.site.qn)
        mps = wl.random_mps(mpo.L, qn, 0, case["m"], seed=int(seed) % (1 << 31))
        return {"case": case, "eng": _engine(mpo, "fp64"), "bonds": mps.bonds, "data": _packed(mps, qn), "L": mpo.L}
    if kind == "regions":
        mpo = _mpo("field")
        qn = list(mpo.site.qn)
        mps = wl.random_mps(mpo.L, qn, 0, 16, seed=int(seed) % (1 << 31))
        eng = _engine(mpo, "bf16", fp64_emulation=True, accurate_edges=2)
        eng.set_mps(mps.bonds, _packed(mps, qn))
        eng.setup_regions(case["regions"], 1, case["m"], **REGION_SWEEP)
        for _ in range(2):
            eng.sweep(case["m"], **REGION_SWEEP)
        return {"case": case, "eng": eng}
    g = _gen(seed)
    if kind == "split":
        mpo = _mpo(case["model"])
        qn = list(mpo.site.qn)
        bonds = _bonds(case["model"], case["m"])
        st = {"case": case, "qn": qn, "bonds": [], "psi": [], "A": [], "B": [], "lam": [], "m": [], "sec": []}
        for j in _split_sites(case):
            bl, bm, br = bonds[j], bonds[j + 1], bonds[j + 2]
            psi = _split_input(g, bl, bm, br, qn, 6.0 if case["mode"] == 2 else 9.0)
            secs = _split_sectors(bl, br, qn)
            rank = {qm: min(sum(bl[q] for q, _ in r), sum(br[q] for _, q in c)) for qm, (r, c) in secs.items()}
            st["bonds"].append(pd.Bond(qn, bl, br, mpo.W[j], mpo.flux[j], mpo.flux[j + 1]))
            st["psi"].append(psi)
            st["m"].append(sum(min(rank[q], bm.get(q, 0)) for q in rank))
            st["sec"].append((bl, br, secs))
            new = functools.partial(torch.zeros, dtype=torch.float64, device="cuda")
            st["A"].append(new(sum(rank[qm] * bl[q] for qm, (r, _) in secs.items() for q, _ in r)))
            st["B"].append(new(sum(rank[qm] * br[q] for qm, (_, c) in secs.items() for _, q in c)))
            st["lam"].append(new(sum(rank.values())))
        return st
    mpo, qn, j, bl, bm, br = _window(case)
    f0, f1, f2 = mpo.flux[j], mpo.flux[j + 1], mpo.flux[j + 2]
    if kind == "env":
        A = _isometry(g, sum(bl.values()), max(bm.values()))     # entries of an isometry's size
        size = sum(bl[q] * bm[q + qn[s]] for q, s in _site_keys(bl, bm, qn))
        A = _randn(g, size) * A.std()
        bond = pd.Bond(qn, bl, bm, mpo.W[j], f0, f1)
        if case["side"] == "left":
            src = _env_input(g, bl, f0, 0)
            out = sum(bm[q] * bm[q - int(f1[w])] for q, w in _env_keys(bm, f1))
        else:
            src = _env_input(g, bm, f1, len(f1) - 1)
            out = sum(bl[q] * bl[q - int(f0[w])] for q, w in _env_keys(bl, f0))
        return {"case": case, "bond": bond, "src": src, "A": A,
                "out": torch.zeros(out, dtype=torch.float64, device="cuda")}
    L = _env_input(g, bl, f0, 0)
    R = _env_input(g, br, f2, len(f2) - 1)
    x = _psi_input(g, bl, br, qn)
    if kind == "heff":
        bond = pd.Bond(qn, bl, br, mpo.W[j], f0, f1, mpo.W[j + 1], f2)
        return {"case": case, "bond": bond, "L": L, "R": R, "x": x, "y": torch.empty_like(x)}
    leaf = [t.requires_grad_() for t in (L, R, x, torch.tensor(mpo.W[j]), torch.tensor(mpo.W[j + 1]))]
    return {"case": case, "static": (qn, bl, br, f0, f1, f2), "leaf": leaf, "ybar": _psi_input(g, bl, br, qn)}


# ------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "heff":
        prec, y = PRECS[case["prec"]], state["y"]
        pd.heff_apply(state["bond"], prec, state["L"].data_ptr(), state["R"].data_ptr(), state["x"].data_ptr(), y.data_ptr())
        return y if case["prec"] == "fp64" else y.float()
    if kind == "env":
        prec, out = PRECS[case["prec"]], state["out"]
        step = pd.env_left if case["side"] == "left" else pd.env_right
        step(state["bond"], prec, state["src"].data_ptr(), state["A"].data_ptr(), out.data_ptr())
        return out if case["prec"] == "fp64" else out.float()
    if kind == "grad":
        from paper_1301_3494_gb300.autograd import heff
        y = heff(*state["static"], *state["leaf"])
        return [y.detach(), *torch.autograd.grad(y, state["leaf"], state["ybar"])]
    if kind == "split":
        ptr = lambda ts: [t.data_ptr() for t in ts]  # noqa: E731
        if case["bonds"] == 1:
            res = [pd.svd_split(state["bonds"][0], state["psi"][0].data_ptr(), state["m"][0], case["mode"],
                                state["A"][0].data_ptr(), state["lam"][0].data_ptr(), state["B"][0].data_ptr())]
        else:
            res = pd.svd_split_batch(state["bonds"], ptr(state["psi"]), state["m"], case["mode"], ptr(state["A"]),
                                     ptr(state["lam"]), ptr(state["B"]))
        out = []
        for b, (mid, trunc) in enumerate(res):
            A, lam, B = state["A"][b], state["lam"][b][: sum(mid.values())], state["B"][b]
            if case["mode"] == 2:
                A, lam, B = A.float(), lam.float(), B.float()
            got = {"kept": np.array(list(mid.values())), "weight": 1.0 - trunc,
                   "psi": _joined(state["sec"][b], state["qn"], mid, A, lam, B)}
            # (an FP32 lambda is the column norms of the very matrices that make psi)
            out.append(got if case["mode"] == 2 else got | {"lam": lam})
        return out
    eng = state["eng"]
    if kind == "sweep":
        eng.set_mps(state["bonds"], state["data"])
        s = eng.sweep(case["m"])
        return {"energy": s["energy"], "lam": [eng.lam(b) for b in range(1, state["L"])]}
    # reduced precision moves the small Schmidt values of a whole sweep: its energy is what is determined
    s = eng.sweep(case["m"], **REGION_SWEEP)
    return {"energy": s["energy"], "steps": s["n_steps"]}


def _joined(sec, qn, mid, A, lam, B):
    """A diag(lambda) B as the flat concatenation of its sector matrices (ascending middle charge,
    rows (q, s1), columns (s2, q_right))."""
    bl, br, secs = sec
    at, off = {}, 0
    for q in bl:
        for s in range(len(qn)):
            if q + qn[s] in mid:
                at[(q, s)] = A[off: off + bl[q] * mid[q + qn[s]]].view(bl[q], -1)
                off += bl[q] * mid[q + qn[s]]
    parts, off, lo = [], 0, 0
    for qm, (rows, cols) in secs.items():
        k = mid.get(qm, 0)
        if not k:
            parts.append(A.new_zeros(sum(bl[q] for q, _ in rows) * sum(br[q] for _, q in cols)))
            continue
        right = []
        for s2, qc in cols:
            right.append(B[off: off + k * br[qc]].view(k, -1))
            off += k * br[qc]
        left = torch.cat([at[r] for r in rows]) * lam[lo: lo + k]
        parts.append((left @ torch.cat(right, 1)).reshape(-1))
        lo += k
    return torch.cat(parts)


# ------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------
def _two_site(W1, W2):
    """Entries (w, s1, s1', s2, s2', w2) that W1 x W2 can produce."""
    return np.argwhere(np.einsum("aijb,bklc->aijklc", np.abs(W1), np.abs(W2), optimize=True) != 0)


def _heff_flops(bl, br, qn, W1, W2, f0, f2):
    ent = _two_site(W1, W2)
    fl, left, right = 0.0, set(), set()
    for q, a, b in _psi_keys(bl, br, qn):
        n = br[q + qn[a] + qn[b]]
        for w, s1, s1p, s2, s2p, w2 in ent:
            if (a, b) != (s1p, s2p) or q + int(f0[w]) not in bl:
                continue
            qo = q + int(f0[w])
            qc = qo + qn[s1] + qn[s2]
            if qc not in br:
                continue
            rows = bl[qo]
            fl += 2.0 * rows * n
            if (q, a, b, w) not in left:
                left.add((q, a, b, w))
                fl += 2.0 * rows * bl[q] * n
            if (qo, s1, s2, w2) not in right:
                right.add((qo, s1, s2, w2))
                fl += 2.0 * rows * n * br[qc]
    return fl


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        # a pair of bond steps per bond, each at least a matvec and a split at dense bond dimension
        m, L = case["m"], case["L"]
        return {"bytes": 8.0 * 2 * L * (2 * m * m * (5 + 4)), "flops": 2.0 * L * (2 * 5 * 8 * m ** 3 / 3.0 + 26.0 * m ** 3)}
    if kind == "regions":
        m = case["m"]
        return {"bytes": 8.0 * 46 * (2 * m * m * (14 + 4)), "flops": 46 * (5 * 2 * 14 * 8 * m ** 3 / 5.0 + 26.0 * m ** 3)}
    if kind == "split":
        bonds = _bonds(case["model"], case["m"])
        qn = list(_mpo(case["model"]).site.qn)
        fl = by = 0.0
        for j in _split_sites(case):
            bl, br = bonds[j], bonds[j + 2]
            for rows, cols in _split_sectors(bl, br, qn).values():
                r, c = sum(bl[q] for q, _ in rows), sum(br[q] for _, q in cols)
                p, n = max(r, c), min(r, c)
                fl += 4.0 * p * n * n + 22.0 * n ** 3
                by += 8.0 * (2 * p * n + (p + n) * n)
        return {"bytes": by, "flops": fl}
    mpo, qn, j, bl, bm, br = _window(case)
    f0, f1, f2 = mpo.flux[j], mpo.flux[j + 1], mpo.flux[j + 2]
    env = lambda b, f: sum(b[q] * b[q - int(f[w])] for q, w in _env_keys(b, f))  # noqa: E731
    if kind == "env":
        site = sum(bl[q] * bm[q + qn[s]] for q, s in _site_keys(bl, bm, qn))
        fl = 0.0
        b0, b1, g0 = (bl, bm, f0) if case["side"] == "left" else (bm, bl, f1)
        sign = 1 if case["side"] == "left" else -1
        nz = np.argwhere(mpo.W[j] != 0)
        used = {(int(e[0] if sign > 0 else e[3]), int(e[2])) for e in nz}
        for q, w in _env_keys(b0, g0):
            k = q - int(g0[w])
            for s in range(len(qn)):
                if (w, s) in used and k + sign * qn[s] in b1:
                    fl += 2.0 * b0[q] * b0[k] * b1[k + sign * qn[s]]
        g1 = f1 if case["side"] == "left" else f0
        for q, w in _env_keys(b1, g1):
            for s in range(len(qn)):
                if q - sign * qn[s] in b0:
                    fl += 2.0 * b1[q] * b1[q - int(g1[w])] * b0[q - sign * qn[s]]
        return {"bytes": 8.0 * (env(bl, f0) + env(bm, f1) + site), "flops": fl}
    psi = sum(bl[q] * br[q + qn[a] + qn[b]] for q, a, b in _psi_keys(bl, br, qn))
    fl = _heff_flops(bl, br, qn, mpo.W[j], mpo.W[j + 1], f0, f2)
    by = 8.0 * (env(bl, f0) + env(br, f2) + 2 * psi)
    if kind == "grad":
        return {"bytes": 3 * by, "flops": 3 * fl}
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------------------
# The same values in 64 bits, plain torch and numpy
# ------------------------------------------------------------------------------------------
def _blocks(flat, keys, rows, cols):
    out, off = {}, 0
    for k in keys:
        r, c = rows(k), cols(k)
        out[k] = flat[off: off + r * c].reshape(r, c)
        off += r * c
    return out


def _exact_heff(qn, bl, br, f0, f2, L, R, x, W12, ent):
    """y = H_eff x; W12 (the two-site operator) may carry gradients."""
    Lb = _blocks(L, _env_keys(bl, f0), lambda k: bl[k[0]], lambda k: bl[k[0] - int(f0[k[1]])])
    Rb = _blocks(R, _env_keys(br, f2), lambda k: br[k[0]], lambda k: br[k[0] - int(f2[k[1]])])
    size = lambda k: br[k[0] + qn[k[1]] + qn[k[2]]]  # noqa: E731
    X = _blocks(x, _psi_keys(bl, br, qn), lambda k: bl[k[0]], size)
    by_in = {}
    for w, s1, s1p, s2, s2p, w2 in ent:
        by_in.setdefault((int(s1p), int(s2p), int(w)), []).append((int(s1), int(s2), int(w2)))
    Y = {}
    for (q, a, b), blk in X.items():
        for w in range(len(f0)):
            lst = by_in.get((a, b, w))
            qo = q + int(f0[w])
            if not lst or (qo, w) not in Lb:
                continue
            LX = Lb[(qo, w)] @ blk
            for s1, s2, w2 in lst:
                qc = qo + qn[s1] + qn[s2]
                if qc not in br or (qc, w2) not in Rb:
                    continue
                Y.setdefault((qo, s1, s2, w2), []).append(W12[w, s1, a, s2, b, w2] * LX)
    out = {k: torch.zeros_like(v) for k, v in X.items()}
    for (qo, s1, s2, w2), terms in Y.items():
        qc = qo + qn[s1] + qn[s2]
        out[(qo, s1, s2)] = out[(qo, s1, s2)] + sum(terms[1:], terms[0]) @ Rb[(qc, w2)].T
    return torch.cat([out[k].reshape(-1) for k in X])


def _exact_env(case, st):
    mpo, qn, j, bl, bm, _ = _window(case)
    f0, f1, W = mpo.flux[j], mpo.flux[j + 1], mpo.W[j]
    A = _blocks(st["A"], _site_keys(bl, bm, qn), lambda k: bl[k[0]], lambda k: bm[k[0] + qn[k[1]]])
    left = case["side"] == "left"
    b0, b1, g0, g1 = (bl, bm, f0, f1) if left else (bm, bl, f1, f0)
    E = _blocks(st["src"], _env_keys(b0, g0), lambda k: b0[k[0]], lambda k: b0[k[0] - int(g0[k[1]])])
    out = {k: torch.zeros(b1[k[0]], b1[k[0] - int(g1[k[1]])], dtype=torch.float64, device="cuda") for k in _env_keys(b1, g1)}
    mixed, half = {}, {}
    for w, s, sp, wp in np.argwhere(W != 0):
        v, wi, wo = float(W[w, s, sp, wp]), int(w if left else wp), int(wp if left else w)
        s, sp = int(s), int(sp)
        for q in b0:
            if (q, wi) not in E:
                continue
            k = q - int(g0[wi])
            bra, ket = ((q, s), (k, sp)) if left else ((q - qn[s], s), (k - qn[sp], sp))
            qo = q + qn[s] if left else q - qn[s]
            if bra not in A or ket not in A or (qo, wo) not in out:
                continue
            if (q, wi, sp) not in half:
                half[(q, wi, sp)] = E[(q, wi)] @ (A[ket] if left else A[ket].T)
            mixed.setdefault((qo, wo, bra), []).append(v * half[(q, wi, sp)])
    for (qo, wo, bra), terms in mixed.items():
        t = sum(terms[1:], terms[0])
        out[(qo, wo)] += (A[bra].T if left else A[bra]) @ t
    return torch.cat([v.reshape(-1) for v in out.values()])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sweep", "regions"):
        return None
    st = prepare(case, seed)
    if kind == "env":
        return _exact_env(case, st)
    if kind == "split":
        return [_exact_split(st, b) for b in range(case["bonds"])]
    mpo, qn, j, bl, bm, br = _window(case)
    f0, f2 = mpo.flux[j], mpo.flux[j + 2]
    W1, W2 = mpo.W[j], mpo.W[j + 1]
    ent = _two_site(W1, W2)
    if kind == "heff":
        W12 = np.einsum("aijb,bklc->aijklc", W1, W2, optimize=True)
        return _exact_heff(qn, bl, br, f0, f2, st["L"], st["R"], st["x"], W12, ent)
    L, R, x, w1, w2 = st["leaf"]
    W12 = torch.einsum("aijb,bklc->aijklc", w1, w2).cuda()
    y = _exact_heff(qn, bl, br, f0, f2, L, R, x, W12, ent)
    got = list(torch.autograd.grad(y, st["leaf"], st["ybar"]))
    got[3], got[4] = got[3] * (w1 != 0), got[4] * (w2 != 0)
    return [y.detach(), *got]


def _exact_split(st, b):
    """Singular values sorted by size over all sectors, the m largest kept and normalised."""
    bl, br, secs = st["sec"][b]
    qn = st["qn"]
    P = _blocks(st["psi"][b], _psi_keys(bl, br, qn), lambda k: bl[k[0]], lambda k: br[k[0] + qn[k[1]] + qn[k[2]]])
    dec = {}
    for qm, (rows, cols) in secs.items():
        M = torch.cat([torch.cat([P[(q, s1, s2)] for s2, _ in cols], 1) for q, s1 in rows])
        dec[qm] = np.linalg.svd(M.cpu().numpy(), full_matrices=False)
    every = np.sort(np.concatenate([s for _, s, _ in dec.values()]))[::-1]
    m = st["m"][b]
    cut = every[m - 1]
    kept = [int(np.sum(s >= cut)) for _, s, _ in dec.values()]
    norm = math.sqrt(float(np.sum(every[:m] ** 2)))
    lam = np.concatenate([s[:k] for (_, s, _), k in zip(dec.values(), kept)]) / norm
    psi = np.concatenate([((u[:, :k] * (s[:k] / norm)) @ v[:k]).reshape(-1) for (u, s, v), k in zip(dec.values(), kept)])
    got = {"psi": torch.from_numpy(psi), "kept": np.array([k for k in kept if k]),
           "weight": float(np.sum(every[:m] ** 2) / np.sum(every ** 2))}
    return got if st["case"]["mode"] == 2 else got | {"lam": torch.from_numpy(lam)}
