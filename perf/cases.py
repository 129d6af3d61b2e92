"""Measured cases of the two-site DMRG hot path.

The cases are the work a program gives this library: the two-site effective Hamiltonian in each
arithmetic (plain FP64, float-float refinement, TF32 and split-BF16 tensor cores, complex and
real), the Lanczos solver, the environment update, whole two-site updates of the
reduced-precision and of the plain FP64 form, and sweeps of a small cylinder. Sizes are those of
the library's own benchmark and tests: Hofstadter cylinders of circumference 4 to 10 at bond
dimensions from tens to 3200, whose charge sectors have very uneven, mostly odd dimensions.

Bond sectors of the H_eff cases follow the recipe of the benchmark (particle number within 3 of
the bond's mean, Gaussian weights, every momentum); sites are in the middle of a ring, where the
MPO bonds are largest. Environments and theta are uniform in [-1, 1) + i [-1, 1) as in the
benchmark's throughput measurement, or, for the solvers, those of a seeded random MPS of the
cylinder, whose H_eff is Hermitian.

The site tensors after an update are defined only up to the phase of each Schmidt vector, so a
program reads an updated state through what does not depend on it: the energy, the discarded
weight, the new bond's charge sectors and its Schmidt values per sector. Updates run a fixed
number of Lanczos steps, so that every pass does the same work.
"""
import ctypes
import functools
import math

import numpy as np
import torch

import paper_1512_03318_gb300 as P

PRECS = {"fp64": P.MRD_PREC_FP64, "tf32": P.MRD_PREC_TF32, "bf16x3": P.MRD_PREC_BF16X3, "ff": P.MRD_PREC_FF}
BASES = {False: P.MRD_BASIS_MIXED, True: P.MRD_BASIS_MIXED_REAL}


def listed():
    return [
        # plain FP64 product of a very small problem (edge bonds, tests): latency and launches
        {"name": "apply_fp64_ly4_chi48", "kind": "apply", "prec": "fp64", "real": False, "ly": 4, "chi": 48},
        # plain FP64 product, the framework's reference form, at an ordinary size
        {"name": "apply_fp64_ly8_chi1024", "kind": "apply", "prec": "fp64", "real": False, "ly": 8, "chi": 1024},
        # split-BF16 product at the headline size: the Lanczos matvec of production updates
        {"name": "apply_bf16x3_ly10_chi3200", "kind": "apply", "prec": "bf16x3", "real": False, "ly": 10, "chi": 3200},
        # TF32 product, the cheaper reduced precision, odd bond dimension
        {"name": "apply_tf32_ly8_chi2049", "kind": "apply", "prec": "tf32", "real": False, "ly": 8, "chi": 2049},
        # split-BF16 product in real arithmetic (the sine / cosine machine)
        {"name": "apply_bf16x3_real_ly6_chi777", "kind": "apply", "prec": "bf16x3", "real": True, "ly": 6, "chi": 777},
        # refinement of a production update: new environments loaded, one float-float product
        {"name": "refine_ff_ly10_chi3200", "kind": "refine", "prec": "ff", "real": False, "ly": 10, "chi": 3200},
        # eigensolver of production updates: split-BF16 matvecs, FP64 Krylov vectors
        {"name": "lanczos_bf16x3_ly8_chi1024", "kind": "lanczos", "prec": "bf16x3", "real": False, "ly": 8, "chi": 1024,
         "steps": 20},
        # eigensolver in plain FP64 on a ragged ordinary problem
        {"name": "lanczos_fp64_ly5_chi301", "kind": "lanczos", "prec": "fp64", "real": False, "ly": 5, "chi": 301,
         "steps": 10},
        # environment update of production updates (both directions), float-float; the new environments
        # are read back, as a program that keeps them on the host does
        {"name": "env_ff_ly8_chi1024", "kind": "env", "prec": "ff", "real": False, "ly": 8, "chi": 1024},
        # whole production update at the headline circumference and bond dimension
        {"name": "update_mixed_ly10_chi3200", "kind": "update", "prec": "bf16x3", "real": False, "ly": 10, "chi": 3200,
         "steps": 20},
        # whole update of the plain FP64 form
        {"name": "update_fp64_ly6_chi512", "kind": "update", "prec": "fp64", "real": False, "ly": 6, "chi": 512,
         "steps": 8},
        # one sweep of a small cylinder (the 4 x 4 cylinder of the tests): tables, launches, host work
        {"name": "sweep_fp64_ly4_chi64", "kind": "sweep", "prec": "fp64", "real": False, "ly": 4, "chi": 64, "steps": 6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "refine", "refine", "lanczos", "env", "update", "sweep"])
    if kind in ("apply", "refine"):
        prec = "ff" if kind == "refine" else rng.choice(["fp64", "bf16x3", "tf32", "bf16x3"])
        ly = rng.choice([4, 5, 6, 8, 10])
        chi = _log_int(rng, 10 * ly, 1024 if prec == "fp64" else 320 * ly)
        real = prec != "fp64" and rng.random() < 0.25
        return {"kind": kind, "prec": prec, "real": real, "ly": ly, "chi": chi}
    if kind == "lanczos":
        return {"kind": kind, "prec": rng.choice(["bf16x3", "tf32", "fp64", "ff"]), "real": False,
                "ly": rng.choice([4, 5, 6]), "chi": _log_int(rng, 50, 500), "steps": rng.randint(4, 20)}
    if kind == "env":
        return {"kind": kind, "prec": rng.choice(["ff", "ff", "fp64"]), "real": False, "ly": rng.choice([4, 5, 6, 8]),
                "chi": _log_int(rng, 50, 1024)}
    if kind == "update":
        prec = rng.choice(["bf16x3", "bf16x3", "fp64"])
        return {"kind": kind, "prec": prec, "real": False, "ly": rng.choice([4, 5, 6, 8]),
                "chi": _log_int(rng, 64, 400 if prec == "fp64" else 1200), "steps": rng.randint(4, 12)}
    return {"kind": kind, "prec": rng.choice(["fp64", "bf16x3"]), "real": False, "ly": rng.choice([3, 4]),
            "chi": _log_int(rng, 16, 200), "steps": rng.randint(3, 6)}


# ---------------------------------------------------------------- problems

@functools.lru_cache(maxsize=None)
def _context():
    return P.Context(0, torch.cuda.current_stream())


@functools.lru_cache(maxsize=None)
def _mpo(lx, ly, real):
    """The model MPO of an lx x ly cylinder with flux 1/ly, t = V = 1."""
    return P.MPO(None, lx, ly, 1, ly, 1.0, 1.0, BASES[real])


def _sectors(chi, ly, n_mean, tag):
    """Bond sectors ((N, K), dim) summing to chi: N within 3 of n_mean, weight exp(-dN^2 / 0.72)
    (1 + u / 4), u uniform in [-1, 1); every sector has at least 4 states when chi allows it."""
    keys = [(n_mean + dn, k) for dn in range(-3, 4) for k in range(ly)]
    least = 4 if chi >= 8 * len(keys) else 0
    u = np.random.RandomState(1000 * ly + tag).uniform(-1.0, 1.0, len(keys))
    w = np.exp(-np.array([(n - n_mean) ** 2 for n, _ in keys]) / 0.72) * (1.0 + 0.25 * u)
    dims = least + np.floor((chi - least * len(keys)) * w / w.sum()).astype(np.int64)
    dims[int(np.argmax(dims))] += chi - int(dims.sum())
    return np.array([[n, k, d] for (n, k), d in zip(keys, dims) if d > 0], dtype=np.int32)


@functools.lru_cache(maxsize=16)
def _problem(ly, chi, real):
    """The description of an H_eff: sectors and MPO of the two sites in the middle of a ring."""
    mpo, site = _mpo(4, ly, real), 2 * ly + ly // 2 - 1
    wi, wj = mpo.site(site), mpo.site(site + 1)
    return {"left": _sectors(chi, ly, 10, 1), "right": _sectors(chi, ly, 10, 2), "m1": site % ly, "m2": (site + 1) % ly,
            "modulus": mpo.modulus, "cl": mpo.bond(site), "cm": mpo.bond(site + 1), "cr": mpo.bond(site + 2),
            "wi_idx": wi[0], "wi_val": wi[1], "wj_idx": wj[0], "wj_val": wj[1]}


def _uniform(n, gen, real):
    x = torch.rand(n, 2, dtype=torch.float64, device="cuda", generator=gen) * 2.0 - 1.0
    if real:
        x[:, 1] = 0.0
    return torch.view_as_complex(x)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _inputs(case, seed, lens):
    g = _generator(seed)
    return [_uniform(n, g, case["real"]) for n in lens]


def _cylinder(case):
    """(lx, particles, centre site) of the cylinder of a state. Short half-filled cylinders give
    the bond dimensions room in the middle of a ring; the sweeps' ly x ly cylinders at one particle
    per ring are those of the tests."""
    ly = case["ly"]
    if case["kind"] == "sweep":
        return ly, ly, 0
    lx = 4 if ly >= 8 else 6
    return lx, lx * ly // 2, (lx // 2) * ly + ly // 2 - 1


def _state(case, seed):
    lx, n, centre = _cylinder(case)
    ly, chi = case["ly"], case["chi"]
    caps = None
    if case["kind"] != "sweep":   # the sector recipe on every bond but the outermost
        caps = [[tuple(int(x) for x in s) for s in _sectors(chi, ly, round(n * j / (lx * ly)), j)]
                if 2 <= j <= lx * ly - 2 else [] for j in range(lx * ly + 1)]
    return P.DMRG(_context(), _mpo(lx, ly, case["real"]), n, 0, chi, seed=1 + int(seed), center=centre, caps=caps)


def _state_problem(case, d):
    """The H_eff of the centre bond of a state: description, environments and a theta length."""
    lx, _, c = _cylinder(case)
    mpo, ly = _mpo(lx, case["ly"], case["real"]), case["ly"]
    wi, wj = mpo.site(c), mpo.site(c + 1)
    prob = {"left": d.bond(c), "right": d.bond(c + 2), "m1": c % ly, "m2": (c + 1) % ly, "modulus": mpo.modulus,
            "cl": mpo.bond(c), "cm": mpo.bond(c + 1), "cr": mpo.bond(c + 2), "wi_idx": wi[0], "wi_val": wi[1],
            "wj_idx": wj[0], "wj_val": wj[1]}
    return prob, [torch.from_numpy(d.env(b, s)).cuda() for b, s in ((c, 0), (c + 2, 1))]


def _params(case):
    fp64 = case["prec"] == "fp64"
    return P.DMRG.params(case["chi"], 1e-14, case["steps"], 0.0, PRECS[case["prec"]], 0 if fp64 else 1, 1e-13)


# ---------------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind, s = case["kind"], {"case": case, "prec": PRECS[case["prec"]]}
    if kind in ("apply", "refine"):
        h = P.Heff(_context(), **_problem(case["ly"], case["chi"], case["real"]))
        if case["real"]:
            h.set_option(P.MRD_OPT_REAL, 1)
        s["h"] = h
        s["l"], s["r"], s["theta"] = _inputs(case, seed, (h.lenv_len, h.renv_len, h.theta_len))
        s["out"] = torch.empty_like(s["theta"])
        h.set_env(s["l"], s["r"])
        return s
    d = _state(case, seed)
    if kind == "lanczos":
        prob, env = _state_problem(case, d)
        d.close()
        s["h"] = P.Heff(_context(), **prob)
        s["h"].set_env(*env)
        s["theta"] = _uniform(s["h"].theta_len, _generator(seed), False)
        return s
    s["d"], s["site"] = d, _cylinder(case)[2]
    if kind == "env":
        # pinned host buffers of the two environments that the updates build
        c = s["site"]
        d.env_update(c, +1, s["prec"])
        d.env_update(c + 1, -1, s["prec"])
        s["host"] = [torch.empty(d.env_len(c + 1, side), dtype=torch.complex128, pin_memory=True) for side in (0, 1)]
    else:
        s["params"] = _params(case)
    return s


def _env_to_host(d, bond, side, host):
    n = ctypes.c_int64()
    d.ctx.check(P.lib().mrd_dmrg_env(d.h, bond, side, ctypes.byref(n),
                                     ctypes.cast(host.data_ptr(), ctypes.POINTER(ctypes.c_double))))
    return host


def _schmidt(d):
    """Charge sectors (N, K) and Schmidt values of the bond the last update cut."""
    b, n = ctypes.c_int32(), ctypes.c_int64()
    d.ctx.check(P.lib().mrd_dmrg_schmidt(d.h, ctypes.byref(b), ctypes.byref(n), None, None))
    nk, v = np.empty((n.value, 2), dtype=np.int32), np.empty(n.value, dtype=np.float64)
    d.ctx.check(P.lib().mrd_dmrg_schmidt(d.h, ctypes.byref(b), ctypes.byref(n),
                                         nk.ctypes.data_as(ctypes.POINTER(ctypes.c_int32)),
                                         v.ctypes.data_as(ctypes.POINTER(ctypes.c_double))))
    return nk, v


def run(s):
    kind = s["case"]["kind"]
    if kind == "apply":
        s["h"].apply(s["theta"], s["out"], s["prec"])
        return s["out"]
    if kind == "refine":
        s["h"].set_env(s["l"], s["r"])
        s["h"].apply(s["theta"], s["out"], s["prec"])
        return s["out"]
    if kind == "lanczos":
        v = s["theta"].clone()
        e, steps = s["h"].lanczos(v, s["case"]["steps"], 0.0, s["prec"])
        return {"energy": e, "steps": steps, "vector": v}
    d, c = s["d"], s["site"]
    if kind == "env":
        d.env_update(c, +1, s["prec"])
        left = _env_to_host(d, c + 1, 0, s["host"][0])
        d.env_update(c + 1, -1, s["prec"])
        return [left, _env_to_host(d, c + 1, 1, s["host"][1])]
    if kind == "update":
        e, discarded = d.update(c, +1, s["params"])
    else:
        e = d.sweep(s["params"])
        discarded = d.stats()[1]
    nk, v = _schmidt(d)
    out = {"energy": e, "sectors": nk, "schmidt": v}
    if kind == "update":
        out["discarded"] = discarded
    return out


# ---------------------------------------------------------------- work

class _Blocks:
    """Charge blocks of an H_eff description: sector lookup, theta blocks and environment blocks
    with their offsets in the flat layouts of the C header."""

    def __init__(self, prob):
        self.mod, self.m = int(prob["modulus"]), (int(prob["m1"]), int(prob["m2"]))
        self.left = [tuple(int(x) for x in s) for s in prob["left"]]
        self.right = [tuple(int(x) for x in s) for s in prob["right"]]
        self.li = {s[:2]: i for i, s in enumerate(self.left)}
        self.ri = {s[:2]: i for i, s in enumerate(self.right)}
        ch = lambda c: [(int(a), int(b) % self.mod) for a, b in c]
        self.cl, self.cm, self.cr = ch(prob["cl"]), ch(prob["cm"]), ch(prob["cr"])
        ent = lambda i, v: [(*(int(x) for x in e), complex(y)) for e, y in zip(i, v)]
        self.wi, self.wj = ent(prob["wi_idx"], prob["wi_val"]), ent(prob["wj_idx"], prob["wj_val"])
        # theta: middle sectors in order; rows (s1, a), columns (s2, b)
        mids = sorted({self.add(q[:2], s, 0) for q in self.left for s in (0, 1)})
        self.theta, self.theta_len = {}, 0     # (a, s1, s2) -> (offset, row stride, b)
        for q in mids:
            rows = [(s, self.li.get(self.add(q, -s, 0))) for s in (0, 1)]
            cols = [(s, self.ri.get(self.add(q, s, 1))) for s in (0, 1)]
            rows, cols = [r for r in rows if r[1] is not None], [c for c in cols if c[1] is not None]
            if not rows or not cols:
                continue
            width, ro = sum(self.right[b][2] for _, b in cols), 0
            for s1, a in rows:
                co = 0
                for s2, b in cols:
                    self.theta[a, s1, s2] = (self.theta_len + ro * width + co, width, b)
                    co += self.right[b][2]
                ro += self.left[a][2]
            self.theta_len += ro * width
        self.lenv, self.lenv_len = self.env(self.left, self.li, self.cl)
        self.renv, self.renv_len = self.env(self.right, self.ri, self.cr)

    def add(self, q, s, site):
        return (q[0] + s, (q[1] + s * self.m[site]) % self.mod)

    def env(self, sec, index, ch):
        out, off = {}, 0                        # (w, sector) -> (offset, image sector)
        for w, c in enumerate(ch):
            for x, q in enumerate(sec):
                y = index.get((q[0] + c[0], (q[1] + c[1]) % self.mod))
                if y is not None:
                    out[w, x] = (off, y)
                    off += q[2] * sec[y][2]
        return out, off

    def pairs(self):
        """MPO pairs (w, w'', s1', s1, s2', s2) -> summed coefficient."""
        by, out = {}, {}
        for w, x, sp, s, v in self.wj:
            by.setdefault(w, []).append((x, sp, s, v))
        for w, x, sp, s, v in self.wi:
            for y, tp, t, u in by.get(x, []):
                k = (w, y, sp, s, tp, t)
                out[k] = out.get(k, 0.0) + v * u
        return out

    def flops(self):
        """Real flops of one product in the order L, W W, R (8 per complex multiply-add)."""
        fl, x, y = 0, {}, set()
        for (a, s1, s2), (_, _, b) in self.theta.items():
            for w in range(len(self.cl)):
                if (w, a) in self.lenv:
                    ap = self.lenv[w, a][1]
                    fl += 8 * self.left[ap][2] * self.left[a][2] * self.right[b][2]
                    x.setdefault((w, s1, s2), []).append((ap, b))
        for w, z, sp, s, tp, t in self.pairs():
            for ap, b in x.get((w, s, t), []):
                fl += 8 * self.left[ap][2] * self.right[b][2]
                y.add((z, ap, sp, tp, b))
        for z, ap, sp, tp, b in y:
            if (z, b) in self.renv:
                fl += 8 * self.left[ap][2] * self.right[b][2] * self.right[self.renv[z, b][1]][2]
        return fl


@functools.lru_cache(maxsize=32)
def _heff_work(ly, chi, real):
    b = _Blocks(_problem(ly, chi, real))
    fl = b.flops()
    return (fl // 4 if real else fl), b.theta_len, b.lenv_len + b.renv_len


def work(case):
    """Bytes: environments, theta and result once each (complex128, or the folded operand's 8 bytes
    per element where the products are reduced-precision). Flops in the definition's order; the
    updates add the Krylov vectors and the block SVD (one Householder bidiagonalisation's worth)."""
    fl, n, env = _heff_work(case["ly"], case["chi"], case["real"])
    kind, wide = case["kind"], case["prec"] in ("fp64", "ff")
    b = (16 if wide else 8) * env
    if kind in ("apply", "refine"):
        return {"bytes": b + 32 * n, "flops": fl}
    if kind == "lanczos":   # every step: the product and the basis read twice for the orthogonalisation
        k = case["steps"]
        return {"bytes": k * (b + 32 * n) + 16 * n * k * k, "flops": k * fl + 8 * n * k * k}
    if kind == "env":       # two environments in, two out; about a quarter of a product each
        return {"bytes": 32 * env, "flops": fl // 2}
    sector = max(1.0, n / max(1, 3 * case["ly"]))
    svd = 16.0 * n * math.sqrt(sector)
    one_b, one_f = case["steps"] * (b + 32 * n) + 32 * env, case["steps"] * fl + fl // 4 + svd
    if kind == "update":
        return {"bytes": one_b, "flops": one_f}
    sites = case["ly"] ** 2
    return {"bytes": 2 * (sites - 1) * one_b / 4, "flops": 2 * (sites - 1) * one_f / 4}


# ---------------------------------------------------------------- exact values

def _product(blk, lenv, renv):
    """theta -> H_eff theta in complex128, by the definition: X_w = L_w theta, the MPO pairs, then R."""
    pairs = {}
    for (w, z, sp, s, tp, t), v in blk.pairs().items():
        if v != 0:
            pairs.setdefault((w, s, t), []).append((z, sp, tp, v))
    dl, dr = [q[2] for q in blk.left], [q[2] for q in blk.right]
    lm = {k: lenv[o: o + dl[k[1]] * dl[y]].view(dl[y], dl[k[1]]) for k, (o, y) in blk.lenv.items()}
    rm = {k: renv[o: o + dr[k[1]] * dr[y]].view(dr[k[1]], dr[y]) for k, (o, y) in blk.renv.items()}

    def view(flat, key):
        off, width, b = blk.theta[key]
        return flat.as_strided((dl[key[0]], dr[b]), (width, 1), off)

    def apply(theta):
        out, y = torch.zeros_like(theta), {}
        for (a, s1, s2), (_, _, b) in blk.theta.items():
            x = view(theta, (a, s1, s2))
            for w in range(len(blk.cl)):
                if (w, a) not in lm:
                    continue
                todo = pairs.get((w, s1, s2))
                if not todo:
                    continue
                xl, ap = lm[w, a] @ x, blk.lenv[w, a][1]
                for z, sp, tp, v in todo:
                    k = (z, ap, sp, tp, b)
                    if k in y:
                        y[k].add_(xl, alpha=v)
                    elif (z, b) in rm:
                        y[k] = v * xl
        for (z, ap, sp, tp, b), x in y.items():
            view(out, (ap, sp, tp)).addmm_(x, rm[z, b])
        return out

    return apply


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply", "refine"):
        blk = _Blocks(_problem(case["ly"], case["chi"], case["real"]))
        lenv, renv, theta = _inputs(case, seed, (blk.lenv_len, blk.renv_len, blk.theta_len))
        return _product(blk, lenv, renv)(theta)
    if kind != "lanczos" or case["chi"] > 1024 or case["steps"] > 20:
        return None
    d = _state(case, seed)                      # the inputs: a random state's environments
    prob, env = _state_problem(case, d)
    d.close()
    blk = _Blocks(prob)
    mv, v = _product(blk, *env), _uniform(blk.theta_len, _generator(seed), False)
    basis, alpha, beta = [v / torch.linalg.vector_norm(v)], [], []
    for j in range(case["steps"]):
        w = mv(basis[j])
        alpha.append(float(torch.vdot(basis[j], w).real))
        q = torch.stack(basis)
        for _ in range(2):
            w = w - (q.conj() @ w) @ q
        beta.append(float(torch.linalg.vector_norm(w)))
        basis.append(w / beta[j])
    k = case["steps"]
    t = np.diag(alpha) + np.diag(beta[:k - 1], 1) + np.diag(beta[:k - 1], -1)
    e, y = np.linalg.eigh(t)
    y = y[:, 0] * np.sign(y[0, 0])
    v = torch.from_numpy(y.astype(np.complex128)).cuda() @ torch.stack(basis[:k])
    return {"energy": float(e[0]), "steps": k, "vector": v / torch.linalg.vector_norm(v)}
