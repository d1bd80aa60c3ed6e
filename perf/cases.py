"""The work this library is used for, as cases that can be timed and compared.

Every case goes through the package's public calls on synthetic silicon
clusters (diamond lattice, jittered by the seed): 10 functions per atom, s
exponents 0.1, 0.3, 1.0, 3.0 and p exponents 0.2, 0.8, a grid of 0.4 bohr
with 6 bohr of vacuum, kT 0.01 Ha unless the case says otherwise; the same
family as the benchmark and the tests.  The kinds:

  dm         density matrix of a given Fock matrix (FP64 or split FP16)
  scf        one SCF cycle of one cluster, split FP16: the whole chain
  batch      one SCF cycle of several ragged clusters together
  density    density of a density matrix on the grid
  potential  matrix of a grid potential
  grid_d     both of these in FP64 with the contracted basis with d shells
  hartree    Kohn-Sham potential and energies of a density
  setup      closed-form integrals and the factorisation for a new geometry
  columns    columns of the density matrix by the sparse-operator route
  train      one training step of the learned warm start

`exact` repeats each in plain torch, FP64, from the formulas.
"""
import math

import numpy as np
import torch

import paper_2108_13478_gb300 as dft
from paper_2108_13478_gb300 import warmstart

SI_A0 = 10.26
DIAMOND = ((0.0, 0.0, 0.0), (0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0),
           (0.25, 0.25, 0.25), (0.25, 0.75, 0.75), (0.75, 0.25, 0.75), (0.75, 0.75, 0.25))
# (l, exponents, coefficients) per shell
SHELLS_SP = ((0, (0.1,), (1.0,)), (0, (0.3,), (1.0,)), (0, (1.0,), (1.0,)), (0, (3.0,), (1.0,)),
             (1, (0.2,), (1.0,)), (1, (0.8,), (1.0,)))
SHELLS_D = ((0, (3.0, 1.0, 0.3), (0.15, 0.55, 0.45)), (0, (0.1,), (1.0,)),
            (1, (0.8, 0.2), (0.4, 0.7)), (2, (0.5,), (1.0,)))
ETA, DEPTH, WIDTH, ION = 1e-10, 4.0, 1.5, 4.0
F64 = torch.float64


def listed():
    return [
        # smallest call: an 8-atom cluster (K = 80), where launches and latency count
        {"name": "dm_fp64_8", "kind": "dm", "atoms": 8, "mixed": False, "tail": 1e-10, "kT": 0.01},
        # the plain FP64 path on a cluster with ragged tiles (K = 370)
        {"name": "dm_fp64_37", "kind": "dm", "atoms": 37, "mixed": False, "tail": 1e-10, "kT": 0.01},
        # the split-FP16 tensor-core path on an ordinary cluster (K = 1230)
        {"name": "dm_mixed_123", "kind": "dm", "atoms": 123, "mixed": True, "tail": 1e-5, "kT": 0.01},
        # the benchmark: one SCF cycle of the 465-atom sphere (K = 4650)
        {"name": "scf_465", "kind": "scf", "atoms": 465, "tail": 1e-5, "pw92": False},
        # a ragged batch of small clusters in one call
        {"name": "batch_8", "kind": "batch", "systems": 8, "atoms_min": 11, "atoms_max": 90, "tail": 1e-5,
         "sizes_seed": 3},
        # collocation and quadrature by themselves, in the mixed path's FP32 arithmetic
        {"name": "density_147", "kind": "density", "atoms": 147, "mixed": True},
        {"name": "potential_147", "kind": "potential", "atoms": 147, "mixed": True},
        # FP64 collocation and quadrature with contracted functions up to d
        {"name": "grid_d_24", "kind": "grid_d", "atoms": 24, "spherical": True},
        # Poisson + LDA with correlation on the benchmark's grid
        {"name": "hartree_465", "kind": "hartree", "atoms": 465, "pw92": True},
        # a new geometry: integrals, Cholesky factor, its inverse
        {"name": "setup_191", "kind": "setup", "atoms": 191, "mixed": True},
        # columns of P by sparse products and PCG
        {"name": "columns_37", "kind": "columns", "atoms": 37, "ncols": 32, "n_cheb": 100, "thresh": 1e-8,
         "kT": 0.1},
        # warm start: loss, gradient and Adam step on one training cluster
        {"name": "train_47", "kind": "train", "atoms": 47},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dm", "dm", "dm", "scf", "batch", "density", "potential", "grid_d", "hartree", "setup",
                       "columns", "train"])
    if kind == "dm":
        mixed = rng.random() < 0.5
        return {"kind": "dm", "atoms": _log(rng, 9, 150) if mixed else _log(rng, 3, 36), "mixed": mixed,
                "tail": rng.choice([1e-5, 1e-6]) if mixed else 1e-10, "kT": rng.choice([0.01, 0.0125, 0.02])}
    if kind == "scf":
        return {"kind": "scf", "atoms": _log(rng, 16, 400), "tail": rng.choice([1e-5, 1e-6]),
                "pw92": rng.random() < 0.5}
    if kind == "batch":
        lo = rng.randint(5, 20)
        return {"kind": "batch", "systems": rng.randint(2, 8), "atoms_min": lo, "atoms_max": lo + rng.randint(10, 60),
                "tail": rng.choice([1e-5, 1e-6]), "sizes_seed": rng.randint(0, 10 ** 6)}
    if kind in ("density", "potential"):
        return {"kind": kind, "atoms": _log(rng, 12, 147), "mixed": rng.random() < 0.75}
    if kind == "grid_d":
        return {"kind": "grid_d", "atoms": _log(rng, 3, 24), "spherical": rng.random() < 0.5}
    if kind == "hartree":
        return {"kind": "hartree", "atoms": _log(rng, 9, 450), "pw92": rng.random() < 0.5}
    if kind == "setup":
        return {"kind": "setup", "atoms": _log(rng, 9, 190), "mixed": rng.random() < 0.5}
    if kind == "columns":
        return {"kind": "columns", "atoms": _log(rng, 8, 36), "ncols": rng.randint(1, 32),
                "n_cheb": rng.randint(20, 100), "thresh": rng.choice([0.0, 1e-8]), "kT": 0.1}
    return {"kind": "train", "atoms": _log(rng, 9, 46)}


# ---- inputs ----

class Cluster:
    """The system description dft.Context reads: n lattice sites nearest to the
    origin, ordered by z, y, x, jittered by the seed; the grid box follows the
    undistorted sites, so that its size does not depend on the seed."""

    def __init__(self, n_atoms, seed, kT=0.01, shells=SHELLS_SP, spherical=True, h=0.4, pad=6.0):
        reach = int(math.ceil((n_atoms * SI_A0 ** 3 / 8 * 3 / (4 * math.pi)) ** (1 / 3) / SI_A0)) + 1
        cells = np.arange(-reach, reach + 1)
        pts = (np.stack(np.meshgrid(cells, cells, cells, indexing="ij"), -1).reshape(-1, 1, 3)
               + np.array(DIAMOND)).reshape(-1, 3) * SI_A0
        pts = pts[np.argsort(np.round((pts ** 2).sum(1), 6), kind="stable")[:n_atoms]]
        pts = pts[np.lexsort((pts[:, 0], pts[:, 1], pts[:, 2]))]
        self.xyz = pts + np.clip(np.random.default_rng([seed, n_atoms]).normal(0.0, 0.05, pts.shape), -0.2, 0.2)
        self.shells, self.spherical, self.n_atoms = shells, spherical, n_atoms
        self.shell_atom = np.repeat(np.arange(n_atoms), len(shells)).astype(np.int32)
        self.shell_l = np.tile([s[0] for s in shells], n_atoms).astype(np.int32)
        self.shell_exp = np.tile([min(s[1]) for s in shells], n_atoms)
        if any(len(s[1]) > 1 for s in shells):
            self.shell_nprim = np.tile([len(s[1]) for s in shells], n_atoms).astype(np.int32)
            self.prim_exp = np.tile(np.concatenate([s[1] for s in shells]), n_atoms)
            self.prim_coef = np.tile(np.concatenate([s[2] for s in shells]), n_atoms)
        lo, hi = pts.min(0) - pad, pts.max(0) + pad
        self.grid_origin, self.grid_h = lo, h
        self.grid_n = np.array([int(math.ceil((hi[d] - lo[d]) / h - 1e-9)) + 1 for d in range(3)])
        self.n_electrons, self.kT = 4.0 * n_atoms, kT
        self.shape = tuple(int(t) for t in self.grid_n[::-1])

    def axes(self):
        return [torch.tensor(self.grid_origin[d] + self.grid_h * np.arange(int(self.grid_n[d])), device="cuda")
                for d in range(3)]


def gaussians(s, amps, width):
    """sum_C amps[C] exp(-|r - R_C|^2 / width^2) on the grid."""
    R = torch.tensor(s.xyz, device="cuda")
    ex, ey, ez = (torch.exp(-((x[None, :] - R[:, d:d + 1]) / width) ** 2) for d, x in enumerate(s.axes()))
    t = (torch.as_tensor(amps, device="cuda", dtype=F64)[:, None, None] * ey[:, :, None]) * ex[:, None, :]
    return (ez.T.contiguous() @ t.reshape(len(R), -1)).reshape(s.shape)


def start_density(s, seed):
    """Superposition of atoms whose charges differ a little, 4 e on average."""
    q = torch.tensor(np.random.default_rng([seed, 7]).normal(0.0, 0.1, s.n_atoms))
    return gaussians(s, (4.0 + q - q.mean()) * (math.pi * WIDTH ** 2) ** -1.5, WIDTH)


def start_potential(s, seed):
    """A screened potential of the wells plus a smooth disturbance."""
    rng = np.random.default_rng([seed, 8])
    return gaussians(s, -DEPTH + rng.normal(0.0, 0.2, s.n_atoms), WIDTH) + gaussians(
        s, 0.5 + rng.normal(0.0, 0.1, s.n_atoms), 3.0)


def distances(R):
    return torch.linalg.norm(R[:, None, :] - R[None, :, :], dim=-1)


def decaying(s, seed):
    """A symmetric matrix that decays with the distance of its atoms, as density matrices do."""
    g = torch.Generator(device="cuda").manual_seed(seed * 1000 + 9)
    R = torch.tensor(s.xyz, device="cuda")
    per = n_functions(s) // s.n_atoms
    d = distances(R).repeat_interleave(per, 0).repeat_interleave(per, 1)
    A = torch.randn(d.shape, generator=g, device="cuda", dtype=F64) * torch.exp(-d / 3.0)
    return (0.1 * (A + A.T) + torch.diag(torch.full((len(d),), 0.5, device="cuda", dtype=F64))).contiguous()


def n_functions(s):
    per = {0: 1, 1: 3, 2: 5 if s.spherical else 6}
    return int(sum(per[int(l)] for l in s.shell_l))


def prec(mixed):
    return dft.DFT_PREC_FP16X3 if mixed else dft.DFT_PREC_FP64


def batch_sizes(case):
    r = np.random.default_rng(case["sizes_seed"])
    lo, hi = math.log(case["atoms_min"]), math.log(case["atoms_max"])
    return [int(round(math.exp(x))) for x in r.uniform(lo, hi, case["systems"])]


def scf_context(s, case):
    ctx = dft.Context(s, precision=prec(True), cheb_tail_tol=case["tail"], model=dft.DFT_MODEL_NEUTRAL,
                      mixer=dft.DFT_MIX_LINEAR, mix_alpha=0.3,
                      xc=dft.DFT_XC_PW92 if case.get("pw92") else dft.DFT_XC_SLATER)
    ctx.overlap_kinetic()
    return ctx


def columns_problem(case, seed):
    """F, mu and the expansion interval of the columns case."""
    s = Cluster(case["atoms"], seed, case["kT"])
    S, T = overlap_kinetic(s)
    F = T + well_matrix(s)
    e = eigen(F, S)[0]
    n_occ = 2 * s.n_atoms
    cols = np.sort(np.random.default_rng([seed, 5]).choice(len(e), min(case["ncols"], len(e)), replace=False))
    mu = float(0.5 * (e[n_occ - 1] + e[n_occ]))
    return s, S, F.contiguous(), [int(c) for c in cols], mu, float(e[0]) - 0.1, float(e[-1]) + 0.1


def prepare(case, seed):
    kind = case["kind"]
    if kind == "dm":
        s = Cluster(case["atoms"], seed, case["kT"])
        ctx = dft.Context(s, precision=prec(case["mixed"]), cheb_tail_tol=case["tail"])
        ctx.overlap_kinetic()
        return {"kind": kind, "ctx": ctx, "F": (overlap_kinetic(s)[1] + well_matrix(s)).contiguous()}
    if kind == "scf":
        s = Cluster(case["atoms"], seed)
        ctx = scf_context(s, case)
        return {"kind": kind, "ctx": ctx, "n": start_density(s, seed), "v": ctx.grid_array(), "P": ctx.matrix()}
    if kind == "batch":
        ss = [Cluster(n, seed + 100 * i) for i, n in enumerate(batch_sizes(case))]
        return {"kind": kind, "ctxs": [scf_context(s, case) for s in ss],
                "n": [start_density(s, seed + i) for i, s in enumerate(ss)]}
    if kind in ("density", "potential"):
        s = Cluster(case["atoms"], seed)
        x = decaying(s, seed) if kind == "density" else start_potential(s, seed)
        return {"kind": kind, "ctx": dft.Context(s, precision=prec(case["mixed"])), "x": x}
    if kind == "grid_d":
        s = Cluster(case["atoms"], seed, shells=SHELLS_D, spherical=case["spherical"], h=0.5, pad=5.0)
        return {"kind": kind, "ctx": dft.Context(s), "v": start_potential(s, seed), "P": decaying(s, seed)}
    if kind == "hartree":
        s = Cluster(case["atoms"], seed)
        ctx = dft.Context(s, model=dft.DFT_MODEL_NEUTRAL, xc=dft.DFT_XC_PW92 if case["pw92"] else dft.DFT_XC_SLATER)
        return {"kind": kind, "ctx": ctx, "n": start_density(s, seed)}
    if kind == "setup":
        return {"kind": kind, "ctx": dft.Context(Cluster(case["atoms"], seed), precision=prec(case["mixed"]))}
    if kind == "columns":
        s, _, F, cols, mu, lo, hi = columns_problem(case, seed)
        ctx = dft.Context(s)
        ctx.overlap_kinetic()
        return {"kind": kind, "ctx": ctx, "args": (F, cols, mu, lo, hi, case["n_cheb"]), "thresh": case["thresh"]}
    s = Cluster(case["atoms"], seed)
    return {"kind": kind, "ctx": dft.Context(s), "ws": warmstart.WarmStart(net_params(seed)),
            "v": (start_potential(s, seed), start_potential(s, seed + 1))}


def run(st):
    kind = st["kind"]
    if kind == "dm":
        P, info = st["ctx"].density_matrix(st["F"])
        return {"P": P, "n_e": info.n_e_trace}
    if kind == "scf":
        n = st["n"].clone()   # the call turns the input density into the next one
        info = st["ctx"].scf_step(n, st["v"], st["P"])
        return {"n": n, "v": st["v"], "P": st["P"], "e": [info.e_total, info.e_kin, info.e_loc, info.n_e_trace]}
    if kind == "batch":
        n = [x.clone() for x in st["n"]]
        infos = dft.dft_scf_step_batched([c.ctx for c in st["ctxs"]], n)
        return {"n": n, "e": [i.e_total for i in infos]}
    if kind == "density":
        return st["ctx"].density_on_grid(st["x"])
    if kind == "potential":
        return st["ctx"].potential_matrix(st["x"])
    if kind == "grid_d":
        return {"V": st["ctx"].potential_matrix(st["v"]), "n": st["ctx"].density_on_grid(st["P"])}
    if kind == "hartree":
        v, e = st["ctx"].hartree_xc(st["n"])
        return {"v": v, "e": list(e)}
    if kind == "setup":
        return list(st["ctx"].overlap_kinetic())
    if kind == "columns":
        return st["ctx"].density_matrix_columns(*st["args"], thresh=st["thresh"], pcg_tol=1e-10)[0]
    ws = st["ws"]
    loss = ws.accumulate(st["ctx"], *st["v"])
    grad = ws.grads()
    ws.adam(1e-3)
    return {"loss": loss, "grad": grad, "params": ws.params()}


# ---- what a pass cannot do without ----

def _tile_pairs(s):
    """512 x sum over grid tiles of (functions that meet the tile)^2."""
    n = [(int(t) + 7) // 8 for t in s.grid_n]
    cnt = np.zeros(n[::-1])
    for l, z, _ in s.shells:
        L, m = half_width(min(z), l), {0: 1, 1: 3, 2: 5 if s.spherical else 6}[l] * len(z)
        for R in s.xyz:
            sl = []
            for d in (2, 1, 0):
                a = max(0, math.ceil((R[d] - L - s.grid_origin[d]) / s.grid_h)) // 8
                b = min(int(s.grid_n[d]) - 1, math.floor((R[d] + L - s.grid_origin[d]) / s.grid_h)) // 8
                sl.append(slice(a, b + 1))
            cnt[tuple(sl)] += m
    return 512.0 * float((cnt ** 2).sum())


def _dm_work(K, tail, kT):
    """A polynomial of degree N takes about 2 sqrt(N) products of symmetric matrices."""
    N = {1e-5: 14.0, 1e-6: 17.0}.get(tail, 29.0) / kT
    return {"bytes": 16.0 * K * K, "flops": 2.0 * math.sqrt(N) * K * K * (K + 1.0)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [work({"kind": "scf", "atoms": n, "tail": case["tail"]}) for n in batch_sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "grid_d":
        s = Cluster(case["atoms"], 0, shells=SHELLS_D, spherical=case["spherical"], h=0.5, pad=5.0)
        K = n_functions(s)
        return {"bytes": 16.0 * (K * K + np.prod(s.shape)), "flops": 2.0 * _tile_pairs(s)}
    s = Cluster(case["atoms"], 0)
    K, G = n_functions(s), float(np.prod(s.shape))
    if kind == "dm":
        return _dm_work(K, case["tail"], case["kT"])
    if kind == "scf":
        w = _dm_work(K, case["tail"], 0.01)
        return {"bytes": 8.0 * (2 * K * K + 3 * G), "flops": w["flops"] + 2.0 * _tile_pairs(s)}
    if kind in ("density", "potential"):
        return {"bytes": 8.0 * (K * K + G), "flops": _tile_pairs(s)}
    if kind == "hartree":
        return {"bytes": 16.0 * G, "flops": 2 * 2.5 * 8 * G * math.log2(8 * G)}
    if kind == "setup":
        return {"bytes": 16.0 * K * K, "flops": 2.0 / 3.0 * K ** 3}
    if kind == "columns":
        return {"bytes": 8.0 * (K * K + K * case["ncols"]), "flops": 2.0 * K * K * case["ncols"] * case["n_cheb"]}
    return {"bytes": 16.0 * G, "flops": 2.0 * 16 * 12 * s.n_atoms * 4.0 / 3.0 * math.pi * (12.0 / 0.4) ** 3 * 0.5}


def tolerance(case):
    """About four times what the start shows against `exact`."""
    kind = case["kind"]
    if kind == "dm":   # FP64: 3000 recurrence steps, 1e-13 seen, more on stiffer overlaps
        return {"rel": 2e-4} if case["mixed"] else {"rel": 1e-11}
    if kind in ("scf", "batch"):
        return {"rel": 2e-4}
    if kind in ("density", "potential"):
        return {"rel": 1.5e-6} if case["mixed"] else {"rel": 1e-12}
    if kind == "columns":   # the threshold and the solver's tolerance
        return {"rel": 1e-6}
    if kind == "train":
        return {"rel": 1e-4, "max": 1e-1}
    return {"rel": 1e-12}


# ---- the same in plain FP64 torch ----

def half_width(zeta, l):
    """L with c(L sqrt(zeta), l) = 1 - ETA."""
    def tail(x):
        if l == 1:
            return math.exp(-x * x)
        return math.erfc(x) + (2 * x * math.exp(-x * x) / math.sqrt(math.pi) if l == 2 else 0.0)
    lo, hi = 0.0, 40.0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if tail(mid) > ETA else (lo, mid)
    return 0.5 * (lo + hi) / math.sqrt(zeta)


def components(l, spherical):
    if l == 0:
        return [[((0, 0, 0), 1.0)]]
    if l == 1:
        return [[((1, 0, 0), 1.0)], [((0, 1, 0), 1.0)], [((0, 0, 1), 1.0)]]
    r3 = math.sqrt(3.0)
    if spherical:   # m = 2, 1, 0, -1, -2 in the order of the library's table
        return [[((2, 0, 0), r3 / 2), ((0, 2, 0), -r3 / 2)], [((1, 1, 0), r3)],
                [((2, 0, 0), -0.5), ((0, 2, 0), -0.5), ((0, 0, 2), 1.0)], [((0, 1, 1), r3)], [((1, 0, 1), r3)]]
    return [[((2, 0, 0), 1.0)], [((0, 2, 0), 1.0)], [((0, 0, 2), 1.0)],
            [((1, 1, 0), 1.0)], [((1, 0, 1), 1.0)], [((0, 1, 1), 1.0)]]


def terms(s):
    """Cartesian terms of all functions: centres, exponents, coefficients, powers, window half-widths, function."""
    def moment(n, p):
        return 0.0 if n % 2 else math.sqrt(math.pi / p) * math.prod(range(1, n, 2)) / (2 * p) ** (n // 2)
    at, z, c, pw, hw, fn, f = [], [], [], [], [], [], 0
    for a in range(s.n_atoms):
        for l, exps, coefs in s.shells:
            L = half_width(min(exps), l)
            for comp in components(l, s.spherical):
                t = [(zz, cc * w * (2 * zz / math.pi) ** 0.75 * (4 * zz) ** (l / 2) / math.sqrt(3.0 if l == 2 else 1.0), p)
                     for zz, cc in zip(exps, coefs) for p, w in comp]
                norm = sum(c1 * c2 * math.prod(moment(p1[d] + p2[d], z1 + z2) for d in range(3))
                           for z1, c1, p1 in t for z2, c2, p2 in t) ** -0.5
                for zz, cc, p in t:
                    at.append(a), z.append(zz), c.append(cc * norm), pw.append(p), hw.append(L), fn.append(f)
                f += 1
    def dev(x):
        return torch.tensor(np.array(x), device="cuda")
    return dict(R=torch.tensor(s.xyz, device="cuda")[dev(at)], z=dev(z), c=dev(c), p=dev(pw), L=dev(hw), f=dev(fn), K=f)


HERMITE = np.polynomial.hermite.hermgauss(5)


def to_functions(t, M):
    if len(t["f"]) == t["K"]:
        return M
    B = torch.zeros(t["K"], len(t["f"]), device="cuda", dtype=F64)
    B[t["f"], torch.arange(len(t["f"]), device="cuda")] = 1.0
    return B @ M @ B.T


def power(x, n):
    return torch.where(n > 0, x, torch.ones_like(x)) * torch.where(n > 1, x, torch.ones_like(x))


def overlap_kinetic(s):
    """S and T in closed form: Gauss-Hermite sums, exact for polynomials times Gaussians."""
    t = terms(s)
    a, b = t["z"][:, None], t["z"][None, :]
    p = a + b
    Sd, Td = [], []
    for d in range(3):
        A, B = t["R"][:, d][:, None], t["R"][:, d][None, :]
        u, v = t["p"][:, d][:, None], t["p"][:, d][None, :]
        E = torch.exp(-a * b / p * (A - B) ** 2) / torch.sqrt(p)
        P = (a * A + b * B) / p
        S1, T1 = torch.zeros_like(p), torch.zeros_like(p)
        for x, w in zip(*HERMITE):
            r = P + x / torch.sqrt(p)
            xa, xb = (r - A).expand_as(p), (r - B).expand_as(p)
            fa, fb = power(xa, u), power(xb, v)
            da = u * power(xa, (u - 1).clamp(min=0)) - 2 * a * xa * fa
            db = v * power(xb, (v - 1).clamp(min=0)) - 2 * b * xb * fb
            S1 += w * fa * fb
            T1 += w * 0.5 * da * db
        Sd.append(S1 * E), Td.append(T1 * E)
    cc = t["c"][:, None] * t["c"][None, :]
    S = cc * Sd[0] * Sd[1] * Sd[2]
    T = cc * (Td[0] * Sd[1] * Sd[2] + Sd[0] * Td[1] * Sd[2] + Sd[0] * Sd[1] * Td[2])
    return to_functions(t, S), to_functions(t, T)


def well_matrix(s):
    """sum_C <a| -DEPTH exp(-|r - R_C|^2 / WIDTH^2) |b> in closed form (s and p functions)."""
    t = terms(s)
    g = 1.0 / WIDTH ** 2
    a, b = t["z"][:, None], t["z"][None, :]
    p = a + b
    q = p + g
    pre = t["c"][:, None] * t["c"][None, :] * (math.pi / q) ** 1.5 * -DEPTH
    geo = []
    for d in range(3):
        A, B = t["R"][:, d][:, None], t["R"][:, d][None, :]
        u, v = t["p"][:, d][:, None] > 0, t["p"][:, d][None, :] > 0
        pre = pre * torch.exp(-a * b / p * (A - B) ** 2)
        geo.append(((a * A + b * B) / p, A, B, u, v, 0.5 * (u & v) / q))
    V = torch.zeros_like(p)
    pg = p * g / q
    for C in torch.tensor(s.xyz, device="cuda"):
        m = torch.ones_like(p)
        r2 = torch.zeros_like(p)
        for d, (P, A, B, u, v, uv) in enumerate(geo):
            Q = (p * P + g * C[d]) / q
            r2 += (P - C[d]) ** 2
            m *= torch.where(u, Q - A, 1.0) * torch.where(v, Q - B, 1.0) + uv
        V += m * torch.exp(-pg * r2)
    return pre * V


def eigen(F, S):
    L = torch.linalg.cholesky(S)
    X = torch.linalg.solve_triangular(L, F, upper=False)
    M = torch.linalg.solve_triangular(L, X.T, upper=False)
    e, U = torch.linalg.eigh(0.5 * (M + M.T))
    return e, torch.linalg.solve_triangular(L.T, U, upper=True)


def density_matrix(F, S, n_e, kT):
    e, C = eigen(F, S)
    def f(mu):
        return 0.5 * (1.0 - torch.tanh(0.5 * (e - mu) / kT))
    lo, hi = float(e[0]) - 40 * kT, float(e[-1]) + 40 * kT
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 2 * float(f(mid).sum()) < n_e else (lo, mid)
    return (C * f(0.5 * (lo + hi))) @ C.T


def slabs(s, t):
    """(planes, Phi[points of the planes, functions]) over the grid, windows applied."""
    tabs = []
    for d, x in enumerate(s.axes()):
        r = x[:, None] - t["R"][:, d][None, :]
        i = torch.arange(len(x), device="cuda")[:, None]
        o, h = s.grid_origin[d], s.grid_h
        inside = (i >= torch.ceil((t["R"][:, d] - t["L"] - o) / h)) & (i <= torch.floor((t["R"][:, d] + t["L"] - o) / h))
        tabs.append(torch.where(inside, power(r, t["p"][:, d][None, :]) * torch.exp(-t["z"] * r * r), 0.0))
    X, Y, Z = tabs[0] * t["c"], tabs[1], tabs[2]
    B = None
    if len(t["f"]) != t["K"]:
        B = torch.zeros(len(t["f"]), t["K"], device="cuda", dtype=F64)
        B[torch.arange(len(t["f"]), device="cuda"), t["f"]] = 1.0
    yx = (Y[:, None, :] * X[None, :, :]).reshape(-1, len(t["f"]))
    for z in range(len(Z)):
        ph = yx * Z[z]
        yield z, ph if B is None else ph @ B


def quadrature(s, v):
    t = terms(s)
    V = torch.zeros(t["K"], t["K"], device="cuda", dtype=F64)
    for z, ph in slabs(s, t):
        V += ph.T @ (v[z].reshape(-1, 1) * ph)
    return V * s.grid_h ** 3


def collocate(s, P):
    t = terms(s)
    n = torch.empty(s.shape, device="cuda", dtype=F64)
    for z, ph in slabs(s, t):
        n[z] = 2.0 * ((ph @ P) * ph).sum(1).reshape(n[z].shape)
    return n


def hartree(s, n, pw92):
    """v_KS of a density with the ionic charges, and h^3 sum v_loc n, the Hartree and the xc energy."""
    h, N = s.grid_h, [2 * t for t in s.shape]
    r2 = 0
    for d in range(3):
        i = torch.arange(N[d], device="cuda", dtype=F64)
        r2 = r2 + (torch.minimum(i, N[d] - i) ** 2).reshape([-1 if k == d else 1 for k in range(3)])
    r = h * torch.sqrt(r2)
    r[0, 0, 0] = h / (3.0 * math.log(2.0 + math.sqrt(3.0)) - 0.5 * math.pi)
    vloc = gaussians(s, [-DEPTH] * s.n_atoms, WIDTH)
    rho = n - gaussians(s, [ION * (math.pi * WIDTH ** 2) ** -1.5] * s.n_atoms, WIDTH)
    vh = torch.fft.irfftn(torch.fft.rfftn(rho, s=N) * torch.fft.rfftn(1.0 / r), s=N)
    vh = h ** 3 * vh[:s.shape[0], :s.shape[1], :s.shape[2]]
    pos = n > 1e-30
    m = torch.where(pos, n, 1.0)
    c = (3.0 * m / math.pi) ** (1.0 / 3.0)
    vx, ex = -c, -0.75 * c
    if pw92:   # Perdew and Wang, Phys. Rev. B 45, 13244 (1992), unpolarised
        A, A1, b1, b2, b3, b4 = 0.031091, 0.21370, 7.5957, 3.5876, 1.6382, 0.49294
        rs = (3.0 / (4.0 * math.pi * m)) ** (1.0 / 3.0)
        sr = torch.sqrt(rs)
        q0 = -2 * A * (1 + A1 * rs)
        q1 = 2 * A * (b1 * sr + b2 * rs + b3 * rs * sr + b4 * rs * rs)
        dq = A * (b1 / sr + 2 * b2 + 3 * b3 * sr + 4 * b4 * rs)
        lg = torch.log1p(1.0 / q1)
        ec = q0 * lg
        vx, ex = vx + ec - rs / 3 * (-2 * A * A1 * lg - q0 * dq / (q1 * q1 + q1)), ex + ec
    vx, ex = torch.where(pos, vx, 0.0), torch.where(pos, ex, 0.0)
    e = [h ** 3 * float((vloc * n).sum()), 0.5 * h ** 3 * float((vh * rho).sum()), h ** 3 * float((ex * n).sum())]
    return vloc + vh + vx, e


def scf_exact(s, n, pw92):
    v, _ = hartree(s, n, pw92)
    S, T = overlap_kinetic(s)
    P = density_matrix(T + quadrature(s, v), S, s.n_electrons, s.kT)
    out = collocate(s, P)
    e_kin = 2.0 * float((P * T).sum())
    e = hartree(s, out, pw92)[1]
    return 0.7 * n + 0.3 * out, v, P, [e_kin + sum(e), e_kin, e[0], s.n_electrons]


def net_params(seed):
    return warmstart.init_params(seed=seed, scale_out=0.5)


def net_exact(s, theta, v_start, v_target):
    """Loss and gradient of the network's potential by autograd, weights rounded to FP16 as the kernels use them."""
    w = torch.tensor(theta, device="cuda").to(torch.float16).to(F64).requires_grad_()
    R = torch.tensor(s.xyz, device="cuda")
    d = distances(R)
    mk = 8.0 * torch.arange(32, device="cuda", dtype=F64) / 31
    near = ((d < 8.0) & (d > 0))[:, :, None]
    G = torch.where(near, torch.exp(-(d[:, :, None] - mk) ** 2 / (2 * (8.0 / 31) ** 2))
                    * 0.5 * (torch.cos(math.pi * d[:, :, None] / 8.0) + 1.0), 0.0).sum(1)
    x, k = G / 4.0, 0
    for o, i in ((128, 32), (128, 128), (128, 128), (16, 128)):
        W, b = w[k:k + o * i].reshape(o, i), w[k + o * i:k + o * i + o]
        k += o * i + o
        x = x @ W.T + b
        if o == 128:
            x = torch.nn.functional.silu(x)
    wk = 0.5 * 6.0 ** (torch.arange(16, device="cuda", dtype=F64) / 15)
    X, Y, Z = s.axes()
    r0 = (v_start - v_target).reshape(len(Z), -1)
    h3 = s.grid_h ** 3
    dc = torch.zeros_like(x)
    loss = 0.0
    c = x.detach()
    for z in range(len(Z)):   # L = h^3 sum (r0 + sum_Ak c_Ak g_Ak)^2 plane by plane
        r2 = ((Z[z] - R[:, 2]) ** 2)[:, None, None] + ((Y[None, :] - R[:, 1:2]) ** 2)[:, :, None] \
            + ((X[None, :] - R[:, 0:1]) ** 2)[:, None, :]
        r2 = r2.reshape(len(R), -1)
        g = [torch.where(r2 < 144.0, torch.exp(-r2 / float(q) ** 2), 0.0) for q in wk]
        res = r0[z] + sum((c[:, q:q + 1] * g[q]).sum(0) for q in range(16))
        loss += h3 * float((res ** 2).sum())
        dc += torch.stack([2 * h3 * (g[q] @ res) for q in range(16)], 1)
    x.backward(dc)
    return loss, w.grad


def exact(case, seed):
    kind = case["kind"]
    if kind == "dm":
        s = Cluster(case["atoms"], seed, case["kT"])
        S, T = overlap_kinetic(s)
        return {"P": density_matrix(T + well_matrix(s), S, s.n_electrons, s.kT), "n_e": s.n_electrons}
    if kind == "scf":
        if case["atoms"] > 100:
            return None
        s = Cluster(case["atoms"], seed)
        n, v, P, e = scf_exact(s, start_density(s, seed), case["pw92"])
        return {"n": n, "v": v, "P": P, "e": e}
    if kind == "batch":
        ns, es = [], []
        for i, m in enumerate(batch_sizes(case)):
            s = Cluster(m, seed + 100 * i)
            n, _, _, e = scf_exact(s, start_density(s, seed + i), False)
            ns.append(n), es.append(e[0])
        return {"n": ns, "e": es}
    if kind in ("density", "potential"):
        s = Cluster(case["atoms"], seed)
        return collocate(s, decaying(s, seed)) if kind == "density" else quadrature(s, start_potential(s, seed))
    if kind == "grid_d":
        s = Cluster(case["atoms"], seed, shells=SHELLS_D, spherical=case["spherical"], h=0.5, pad=5.0)
        return {"V": quadrature(s, start_potential(s, seed)), "n": collocate(s, decaying(s, seed))}
    if kind == "hartree":
        s = Cluster(case["atoms"], seed)
        v, e = hartree(s, start_density(s, seed), case["pw92"])
        return {"v": v, "e": e}
    if kind == "setup":
        return list(overlap_kinetic(Cluster(case["atoms"], seed)))
    if kind == "columns":
        s, S, F, cols, mu, lo, hi = columns_problem(case, seed)
        e, C = eigen(F, S)
        N = case["n_cheb"]
        th = math.pi * (np.arange(4 * N) + 0.5) / (4 * N)
        fk = 0.5 * (1 - np.tanh(0.5 * (0.5 * (hi + lo) + 0.5 * (hi - lo) * np.cos(th) - mu) / s.kT))
        a = np.array([(1 if l == 0 else 2) / (4 * N) * np.sum(fk * np.cos(l * th)) for l in range(N)])
        x = (e.cpu().numpy() - 0.5 * (hi + lo)) / (0.5 * (hi - lo))
        f = torch.tensor(np.polynomial.chebyshev.chebval(x, a), device="cuda")
        return ((C * f) @ C.T)[:, cols]
    s = Cluster(case["atoms"], seed)
    loss, grad = net_exact(s, net_params(seed), start_potential(s, seed), start_potential(s, seed + 1))
    return {"loss": loss, "grad": grad, "params": None}
