"""Benchmark: SCF steps of the Chebyshev density-matrix DFT on one GB300.

A step is one full SCF cycle through the C ABI (dft_scf_step): Hartree +
LDA potential, quadrature into the Fock matrix, spectral bounds, Chebyshev
moments, mu, the Chebyshev density matrix, collocation of n(r), the energy
and the density mixing.  The metric is P-columns/s: basis functions (columns
of P) produced per second of SCF wall time, with the SCF-step time beside it.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME]
                  [--precision fp64|bf16x3] [--impl ours|reference]

--impl reference times the FP64 CPU oracle (the reference arm of this
repository) on a bounded sample of the same workload.  Under torchrun every
rank runs an independent replica (the path has no cross-GPU exchange here);
rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "P-columns/s & SCF-step time, mixed vs FP64 GPU at <=1e-5 Ha/atom error"
PEAKS_PATH = os.path.join(ROOT, "MEASURED_PEAKS.json")
# FP64 issue rate of GB300: 1.25 TFLOP/s nominal over 152 SMs at 2.07 GHz
# is 2 DFMA per SM per clock
FP64_FLOP_PER_SM_CLK = 4.0
N_SM = 152


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--workload", default="sphere25")
    ap.add_argument("--precision", default="fp16x3", choices=["fp64", "fp16x3", "bf16x3"])
    ap.add_argument("--dm-only", action="store_true",
                    help="time one dft_density_matrix call on the start potential instead of SCF steps")
    ap.add_argument("--no-compare", action="store_true",
                    help="skip the mixed-vs-FP64 comparison on the 64-atom cluster")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--model", default="neutral", choices=["neutral", "literal"])
    ap.add_argument("--mixer", default="pulay", choices=["pulay", "kerker", "linear"],
                    help="density mixing (linear 0.3 diverges for the neutral model on the R = 25 sphere)")
    ap.add_argument("--cheb-tail", type=float, default=None,
                    help="tail tolerance that fixes the Chebyshev order N_C (default: 1e-10 for fp64, "
                         "1e-5 for the mixed precisions)")
    ap.add_argument("--cpu-budget", type=float, default=20.0, help="seconds of oracle work for cpu_baseline")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sparse", action="store_true",
                    help="skip the sparse-operator route's sub-record (dft_density_matrix_columns)")
    ap.add_argument("--no-reuse-mu", action="store_true",
                    help="mixed precisions: run the moments pass on every SCF cycle (default: skip it while mu "
                         "has settled)")
    ap.add_argument("--time-to-solution", action="store_true",
                    help="instead of the step benchmark: converged SCF of the ragged batch tiny8 + tiny37 + "
                         "cluster64 with the FP64 GPU path (one system at a time) and with the mixed, batched, "
                         "warm-started path, wall time against the oracle's converged energies")
    ap.add_argument("--accuracy-workload", default="sphere40",
                    help="workload of the one-density-matrix accuracy record against the oracle's exact traces "
                         "(tests/golden/dm_<name>.json); 'none' leaves it out")
    return ap.parse_args()


def cheb_tail(args):
    """Tail tolerance of the Chebyshev order: sum_{l >= N_C} |a_l| < tol.  The
    FP64 path keeps 1e-10 (P to 1e-9).  The mixed path takes 1e-5: measured
    with the oracle (truncated against exact Fermi-Dirac density matrix, same
    padded bounds), the truncation error is 1.1e-8 Ha/atom on the 64-atom
    cluster and 9e-10 on the 465-atom sphere, two orders below what the
    split-FP16 products already cost (2-4e-6 Ha/atom), for 17% fewer
    recurrence steps than 1e-6 and half those of 1e-10."""
    if args.cheb_tail is not None:
        return args.cheb_tail
    return 1e-10 if args.precision == "fp64" else 1e-5


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except FileNotFoundError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        return self.summarise(self.lines)

    @staticmethod
    def summarise(lines):
        """Median SM clock, the largest maximum clock and every throttle reason
        seen Active over the samples (CSV rows in the order of Q; rows that
        are short or carry no number, such as "[N/A]", are skipped)."""
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": sorted(reasons), "samples": len(sm)}


def peaks():
    try:
        return json.load(open(PEAKS_PATH))
    except Exception:
        return {}


def tc_tiles(K, bm=128, bn=256):
    """Output tiles of the tensor-core step that reach the upper triangle."""
    mt, nt = -(-K // bm), -(-K // bn)
    return sum(1 for i in range(mt) for j in range(nt) if j * bn + bn - 1 >= i * bm)


def cpu_baseline(sysm, budget_s):
    """The FP64 oracle, as it stands, on a bounded sample of one SCF step:
    the eigensolve-based DM and the Poisson solve in full, quadrature and
    collocation on a slab of z-planes scaled to the whole grid (their cost is
    uniform per plane), the eigensolve scaled by K^3 when K is too large."""
    import scipy.linalg as sla  # noqa: F401
    from oracle import basis, dm, grid_ops, poisson, scf
    import oracle.grid_ops as go
    t0 = time.perf_counter()
    st = scf.setup(sysm)
    n0 = scf.ion_density(sysm)
    v, _, _ = scf.potential(st, n0)
    t_pois = 0.0
    a = time.perf_counter()
    poisson.hartree(sysm, n0, st.c0)
    t_pois = time.perf_counter() - a
    nz = int(sysm.grid_n[2])
    per_plane = sysm.n_basis * int(sysm.grid_n[0]) * int(sysm.grid_n[1])
    planes = max(1, min(nz, int(2e8 // max(1, per_plane * 8)) or 1))
    planes = min(planes, 8)
    sub = type(sysm)(**{**sysm.__dict__})
    sub.grid_n = np.array([sysm.grid_n[0], sysm.grid_n[1], planes])
    a = time.perf_counter()
    go.potential_matrix(sub, v[:planes], st.model.eta)
    t_quad = (time.perf_counter() - a) * nz / planes
    K = sysm.n_basis
    P = np.eye(K) * 0.01
    a = time.perf_counter()
    go.density_on_grid(sub, P, st.model.eta)
    t_col = (time.perf_counter() - a) * nz / planes
    F = st.T + np.diag(np.diag(st.S))
    ks = min(K, 1500)
    a = time.perf_counter()
    dm.dm_exact(F[:ks, :ks] + st.T[:ks, :ks], st.S[:ks, :ks], min(sysm.n_electrons, ks), 1.0 / sysm.kT)
    t_eig = (time.perf_counter() - a) * (K / ks) ** 3
    t_step = t_pois * 2 + t_quad + t_col + t_eig
    return {"value": K / t_step, "unit": "P-columns/s", "cores": os.cpu_count(), "kind": "oracle",
            "sample": (f"{sysm.name} SCF step: eigensolve DM ({'full' if ks == K else f'K={ks}, x K^3'}), "
                       f"2 Poisson, quadrature+collocation on {planes}/{nz} planes (x planes)"),
            "projected_step_s": t_step,
            "seconds": time.perf_counter() - t0, "stage_s": {"eig": t_eig, "quad": t_quad, "coll": t_col,
                                                             "poisson": 2 * t_pois}}


def run_batched(args, rank, world):
    """Ragged batch: every SCF step advances all systems with one
    dft_scf_step_batched call (the products of all systems' expansions merged
    into tensor-core launches).  Value = sum of K over systems x steps / time."""
    import torch
    import torch.distributed as dist
    import paper_2108_13478_gb300 as dft
    import workloads as w
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl")
    systems = w.config_batch(args.workload)
    prec = {"fp16x3": dft.DFT_PREC_FP16X3, "bf16x3": dft.DFT_PREC_BF16X3}[args.precision]
    # the largest system leads (its workspace holds the batch tables)
    order = sorted(range(len(systems)), key=lambda i: -systems[i].n_basis)
    ctxs = []
    for i in order:
        c = dft.Context(systems[i], device=f"cuda:{local}", precision=prec, cheb_tail_tol=cheb_tail(args), mix_alpha=0.3,
                        mixer=dft.DFT_MIX_PULAY, kerker_q0=0.8, mix_history=8, model=dft.DFT_MODEL_NEUTRAL)
        c.overlap_kinetic()
        ctxs.append(c)
    dens = [c.initial_density() for c in ctxs]
    handles = [c.ctx for c in ctxs]
    for _ in range(args.warmup):
        dft.dft_scf_step_batched(handles, dens)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    sampler = ClockSampler(local)
    sampler.start()
    l0 = dft.dft_kernel_launches()
    ms = []
    infos = None
    for _ in range(args.steps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        infos = dft.dft_scf_step_batched(handles, dens)
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
    launches = (dft.dft_kernel_launches() - l0) / args.steps
    clocks = sampler.stop()
    total_ms = max_over_ranks(sum(ms), world, f"cuda:{local}")
    ksum = sum(c.K for c in ctxs)
    value = job_throughput(world, ksum, args.steps, total_ms)
    n_c = [i.n_cheb for i in infos]
    line = {"metric": METRIC, "value": value, "unit": "P-columns/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": args.precision, "data": "synthetic",
            "config": {"workload": args.workload, "systems": len(ctxs), "sum_n_basis": ksum,
                       "cheb_tail_tol": cheb_tail(args),
                       "n_basis_range": [min(c.K for c in ctxs), max(c.K for c in ctxs)],
                       "n_cheb_range": [min(n_c), max(n_c)], "model": "neutral",
                       "mixer": "pulay alpha 0.3 kerker q0 0.8 hist 8", "batched": "dft_scf_step_batched",
                       "l2": "working set above L2 (sum of operands)", "parallelism": f"replicas x{world}"},
            "gpu_launches": int(launches), "clocks": clocks,
            "stages_ms": [round(x, 3) for x in infos[0].ms_stage]}
    if rank == 0:
        print(json.dumps(line), flush=True)
    for c in ctxs:
        c.close()
    if world > 1:
        dist.destroy_process_group()


def run_dm_only(args, dft, torch, sysm, prec, local, rank):
    """P-columns/s of dft_density_matrix alone (K / its wall time), on the
    Fock matrix of the superposition-of-atoms start; for workloads where a
    full SCF step is minutes long (the 1963-atom sphere)."""
    t0 = time.perf_counter()
    ctx = dft.Context(sysm, device=f"cuda:{local}", precision=prec, cheb_tail_tol=cheb_tail(args),
                      model=dft.DFT_MODEL_NEUTRAL)
    ctx.overlap_kinetic()
    n0 = ctx.initial_density()
    v, _ = ctx.hartree_xc(n0)
    V = ctx.potential_matrix(v)
    S, T = ctx.overlap_kinetic()
    F = V + T
    torch.cuda.synchronize()
    setup_s = time.perf_counter() - t0
    ms, infos = [], []
    for _ in range(args.steps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        _, info = ctx.density_matrix(F)
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
        infos.append(info)
    K = ctx.K
    t = statistics.median(ms)
    info = infos[-1]
    line = {"metric": METRIC, "value": K / (t / 1000.0), "unit": "P-columns/s (dft_density_matrix)", "n_gpus": 1,
            "steps": args.steps, "warmup": 0, "ms_per_step": t, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": args.precision, "data": "synthetic",
            "config": {"workload": sysm.name, "n_basis": K, "n_atoms": sysm.n_atoms, "kT": sysm.kT,
                       "n_cheb": info.n_cheb, "cheb_tail_tol": cheb_tail(args), "mode": "density matrix only",
                       "setup_s": setup_s},
            "stages_ms": [round(x, 3) for x in info.ms_stage],
            "roofline": expansion_roofline(infos, K, False, *tensor_peak(peaks()))}
    if rank == 0:
        print(json.dumps(line), flush=True)
    ctx.close()


def dm_accuracy(dft, torch, local, name, tail):
    """One mixed-precision dft_density_matrix at the workload's own size,
    timed with CUDA events, against the oracle's exact density-matrix traces
    (tests/golden/dm_<name>.json, written by tests/golden/make_dm_golden.py
    from one generalised eigensolve).  The Fock matrix is the golden's,
    F = T + V[v_loc]: T from the closed-form kernel, V the FP64 quadrature of
    v_loc (the potential of an electron-free literal-model context), built
    with the library and checked against the golden's fingerprints before
    use.  The energy errors per atom are reported with the FP64
    electron-count correction and, through the band-energy shift the library
    reports for it, without it (band energy)."""
    import workloads as w
    path = os.path.join(ROOT, "tests", "golden", f"dm_{name}.json")
    if not os.path.exists(path):
        return {"workload": name, "skipped": "no oracle golden traces"}
    g = json.load(open(path))
    s = w.config_system(name)
    dev = f"cuda:{local}"
    t0 = time.perf_counter()
    c64 = dft.Context(s, device=dev, precision=dft.DFT_PREC_FP64, model=dft.DFT_MODEL_LITERAL)
    v, _ = c64.hartree_xc(c64.grid_array())          # n = 0: v_KS = v_loc
    V = c64.potential_matrix(v)
    c64.close()
    del v, c64
    ctx = dft.Context(s, device=dev, precision=dft.DFT_PREC_FP16X3, cheb_tail_tol=tail, model=dft.DFT_MODEL_NEUTRAL)
    S, T = ctx.overlap_kinetic()
    F = V
    F += T
    torch.cuda.synchronize()
    setup_s = time.perf_counter() - t0
    fp = g["fingerprint"]
    fp_err = max(abs(float(torch.trace(F)) - fp["trace_F"]) / abs(fp["trace_F"]),
                 abs(float(torch.linalg.norm(F)) - fp["frob_F"]) / fp["frob_F"],
                 abs(float(torch.linalg.norm(S)) - fp["frob_S"]) / fp["frob_S"])
    out = {"workload": name, "n_basis": s.n_basis, "n_atoms": s.n_atoms, "kT": s.kT, "cheb_tail_tol": tail,
           "precision": "fp16x3", "setup_s": round(setup_s, 2), "fock_fingerprint_rel_err": fp_err}
    if fp_err > 1e-9:
        out["skipped"] = "Fock matrix differs from the golden's"
        ctx.close()
        return out
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    P, info = ctx.density_matrix(F)
    e1.record(stream)
    e1.synchronize()
    ms = e0.elapsed_time(e1)
    K, na = s.n_basis, s.n_atoms
    e_kin = 2.0 * float(torch.sum(P * T))
    e_band = 2.0 * float(torch.sum(P * F))
    n_e = 2.0 * float(torch.sum(P * S))
    out.update({
        "ms": ms, "value": K / (ms / 1000.0), "unit": "P-columns/s (dft_density_matrix)", "n_cheb": info.n_cheb,
        "stages_ms": [round(x, 3) for x in info.ms_stage],
        "dE_kin_per_atom": abs(e_kin - g["e_kin"]) / na, "dE_band_per_atom": abs(e_band - g["e_band"]) / na,
        "dE_band_per_atom_uncorrected": abs(e_band - info.e_band_correction - g["e_band"]) / na,
        "n_e_trace": n_e, "n_e_uncorrected": info.n_e_uncorrected, "n_electrons": s.n_electrons,
        "mu": info.mu, "mu_oracle": g["mu"], "mu_correction": info.mu_correction,
        "gate_1e-5_Ha_per_atom": bool(abs(e_kin - g["e_kin"]) / na <= 1e-5 and abs(e_band - g["e_band"]) / na <= 1e-5),
        "roofline": expansion_roofline([info], K, False, *tensor_peak(peaks())),
        "reference": "oracle exact traces, tests/golden/" + os.path.basename(path)})
    ctx.close()
    return out


TTS_NAMES = ("tiny8", "tiny37", "cluster64")


def time_to_solution(args, dft, torch, local):
    """Wall time of converged SCF runs on a ragged batch of three clusters
    (K = 80, 370, 640) whose converged energies the oracle wrote
    (tests/golden/scf_<name>.json): the FP64 GPU path one system at a time,
    against the mixed path (split FP16, Chebyshev tail 1e-6, mu reuse) with
    all three systems in dft_scf_step_batched, started from the learned warm
    start (network trained here on eight R = 6-9 bohr spheres, training time
    reported apart) and from the atomic start.  A run stops when every system
    meets |dE|/atom < 1e-7 between cycles and max|n_out - n_in| < 1e-5; its
    energies must be within 1e-5 Ha/atom of the oracle's.  Times are CUDA
    events around each SCF call (and the warm start's first half-cycle)."""
    import workloads as w
    from paper_2108_13478_gb300 import warmstart as ws_mod
    dev = f"cuda:{local}"
    gold = {}
    for n in TTS_NAMES:
        g = json.load(open(os.path.join(ROOT, "tests", "golden", f"scf_{n}.json")))
        gold[n] = g["E_per_atom"]
    systems = [w.config_system(n) for n in TTS_NAMES]
    common = dict(model=dft.DFT_MODEL_NEUTRAL, mixer=dft.DFT_MIX_PULAY, mix_alpha=0.3, kerker_q0=0.8, mix_history=8)

    def ev():
        return torch.cuda.Event(enable_timing=True)

    def converged(info, it):
        return it > 0 and abs(info.de_per_atom) < 1e-7 and info.residual < 1e-5
    out = {"systems": list(TTS_NAMES), "n_basis": [s.n_basis for s in systems], "stop": "|dE|/atom < 1e-7 and "
           "max|n_out - n_in| < 1e-5", "reference": "oracle converged energies, tests/golden/scf_<name>.json"}
    # FP64 GPU, one system at a time
    fp64 = {"seconds": 0.0, "cycles": [], "dE_per_atom": []}
    for s, n in zip(systems, TTS_NAMES):
        ctx = dft.Context(s, device=dev, precision=dft.DFT_PREC_FP64, cheb_tail_tol=1e-10, **common)
        ctx.overlap_kinetic()
        dens = ctx.initial_density()
        for it in range(150):
            e0, e1 = ev(), ev()
            e0.record()
            info = ctx.scf_step(dens)
            e1.record()
            e1.synchronize()
            fp64["seconds"] += e0.elapsed_time(e1) / 1000.0
            if converged(info, it):
                break
        fp64["cycles"].append(it + 1)
        fp64["dE_per_atom"].append(abs(info.e_total / s.n_atoms - gold[n]))
        ctx.close()
    out["fp64_one_by_one"] = fp64
    # the learned warm start, trained on other clusters
    t0 = time.perf_counter()
    radii = np.random.default_rng(77).uniform(6.0, 9.0, 8)
    train = [w.config_system(f"sphereR{r:.3f}", seed=700 + i) for i, r in enumerate(radii)]
    data = ws_mod.training_set(train, cheb_tail_tol=1e-6, reuse_mu=1)
    net = ws_mod.WarmStart(ws_mod.init_params(seed=1), device=dev)
    hist = ws_mod.train(net, data, epochs=120, lr=3e-3)
    for c, _, _ in data:
        c.close()
    out["warm_start_training"] = {"spheres": len(train), "radii": [round(float(r), 3) for r in radii],
                                  "epochs": 120, "loss_first": hist[0], "loss_last": hist[-1],
                                  "seconds": time.perf_counter() - t0}
    for key, warm in (("mixed_batched_warm", True), ("mixed_batched_atoms", False)):
        ctxs = [dft.Context(s, device=dev, precision=dft.DFT_PREC_FP16X3, cheb_tail_tol=1e-6, reuse_mu=1,
                            **common) for s in systems]
        for c in ctxs:
            c.overlap_kinetic()
        rec = {"seconds": 0.0, "cycles": [None] * len(ctxs), "dE_per_atom": [None] * len(ctxs)}
        e0, e1 = ev(), ev()
        e0.record()
        dens = []
        for c in ctxs:
            v0 = ws_mod.start_potential(c)
            if warm:
                v0 = net.potential(c, v0)
                n1 = c.grid_array()
                dft.dft_density_from_potential(c.ctx, v0, n1)
                dens.append(n1)
            else:
                dens.append(c.initial_density())
        e1.record()
        e1.synchronize()
        rec["seconds"] += e0.elapsed_time(e1) / 1000.0
        for it in range(150):
            e0, e1 = ev(), ev()
            e0.record()
            infos = dft.dft_scf_step_batched([c.ctx for c in ctxs], dens)
            e1.record()
            e1.synchronize()
            rec["seconds"] += e0.elapsed_time(e1) / 1000.0
            for q, (info, s, n) in enumerate(zip(infos, systems, TTS_NAMES)):
                if rec["cycles"][q] is None and converged(info, it):
                    rec["cycles"][q] = it + 1
                    rec["dE_per_atom"][q] = abs(info.e_total / s.n_atoms - gold[n])
            if all(cq is not None for cq in rec["cycles"]):
                break
        out[key] = rec
        for c in ctxs:
            c.close()
    ok = all(d is not None and d <= 1e-5 for k in ("mixed_batched_warm", "mixed_batched_atoms")
             for d in out[k]["dE_per_atom"]) and all(d <= 1e-5 for d in fp64["dE_per_atom"])
    out["gate_1e-5_Ha_per_atom"] = ok
    out["speedup_vs_fp64"] = {k: fp64["seconds"] / out[k]["seconds"] for k in ("mixed_batched_warm",
                                                                                 "mixed_batched_atoms")}
    return out


def compare_precisions(dft, torch, local, tail, name="cluster64", steps=2):
    """Mixed (FP16x3) and FP64 GPU paths on the same SCF steps of the 64-atom
    cluster (the largest case where the FP64 path finishes in seconds), both
    with the same Chebyshev tail tolerance: step time of each and the energy
    difference per atom."""
    import workloads as w
    sysm = w.config_system(name)
    out = {"workload": name, "n_basis": sysm.n_basis, "steps": steps, "cheb_tail_tol": tail}
    res = {}
    for prec, key in ((dft.DFT_PREC_FP64, "fp64"), (dft.DFT_PREC_FP16X3, "fp16x3")):
        ctx = dft.Context(sysm, device=f"cuda:{local}", precision=prec, cheb_tail_tol=tail, mix_alpha=0.3,
                          mixer=dft.DFT_MIX_PULAY, kerker_q0=0.8, mix_history=8, model=dft.DFT_MODEL_NEUTRAL)
        ctx.overlap_kinetic()
        n = ctx.initial_density()
        ms, es = [], []
        for _ in range(steps):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            info = ctx.scf_step(n)
            e1.record()
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
            es.append(info.e_total / sysm.n_atoms)
        res[key] = (ms, es)
        ctx.close()
    out["fp64_ms_per_step"] = statistics.median(res["fp64"][0])
    out["fp16x3_ms_per_step"] = statistics.median(res["fp16x3"][0])
    out["speedup"] = out["fp64_ms_per_step"] / out["fp16x3_ms_per_step"]
    out["max_abs_dE_per_atom"] = max(abs(a - b) for a, b in zip(res["fp64"][1], res["fp16x3"][1]))
    return out


def sparse_route(dft, torch, local, tail, sm_mhz, name="cluster64", ncols=32, thresh=1e-8):
    """The sparse-operator route (dft_density_matrix_columns) on the 64-atom
    cluster: one block of columns P u_alpha by the vector recurrence with
    block-Jacobi PCG solves on S and F without their entries below 1e-8, at
    the mu, bounds and N_C of the FP64 dense route on the same Fock matrix.
    P-columns/s, solver work, the FP64 rate of the sparse products (the
    route's arithmetic) and the largest difference from the dense route's
    columns."""
    import workloads as w
    sysm = w.config_system(name)
    ctx = dft.Context(sysm, device=f"cuda:{local}", precision=dft.DFT_PREC_FP64, cheb_tail_tol=tail,
                      model=dft.DFT_MODEL_NEUTRAL)
    _, T = ctx.overlap_kinetic()
    v, _ = ctx.hartree_xc(ctx.initial_density())
    F = (ctx.potential_matrix(v) + T).contiguous()
    P, info = ctx.density_matrix(F)
    K = ctx.K
    cols = [int(x) for x in np.linspace(0, K - 1, ncols).round()]
    out, ci = ctx.density_matrix_columns(F, cols, info.mu, info.e_min, info.e_max, info.n_cheb, thresh=thresh,
                                         pcg_tol=1e-10)
    torch.cuda.synchronize()
    dev = float((out - P[:, cols]).abs().max() / P.abs().max())
    t = ci.ms / 1000.0
    # sparse products: S p in every PCG iteration of the slowest column, F U once per step
    flops = 2.0 * ncols * (ci.nnz_s * ci.pcg_iterations + ci.nnz_f * (info.n_cheb - 1))
    peak = FP64_FLOP_PER_SM_CLK * N_SM * sm_mhz * 1e6 / 1e12
    ctx.close()
    return {"workload": name, "n_basis": K, "columns": ncols, "n_cheb": info.n_cheb, "value": ncols / t,
            "unit": "P-columns/s (dft_density_matrix_columns)", "ms": ci.ms, "precond": "block-Jacobi",
            "thresh": thresh, "pcg_tol": 1e-10, "pcg_iterations": ci.pcg_iterations, "pcg_solves": ci.pcg_solves,
            "iterations_per_solve": ci.pcg_iterations / max(1, ci.pcg_solves), "not_converged": ci.not_converged,
            "nnz_s": ci.nnz_s, "nnz_f": ci.nnz_f, "max_rel_dev_from_dense": dev,
            "roofline": {"kernel": "k_spmm", "bound": "alu", "achieved": flops / t / 1e12, "peak": peak,
                         "unit": "TFLOP/s", "frac": flops / t / 1e12 / peak,
                         "note": "whole-call time; FP64 issue rate 4 flop/SM/clk x 152 SMs x median SM clock"}}


def run_reference_batch(args, rank):
    """Oracle on a bounded sample of a ragged batch: the bounded one-step
    sample (cpu_baseline) of 8 systems spread over the size range, scaled to
    the whole batch by the number of systems."""
    if rank != 0:
        return
    import workloads as w
    systems = sorted(w.config_batch(args.workload), key=lambda s: s.n_basis)
    pick = [systems[i] for i in np.linspace(0, len(systems) - 1, min(8, len(systems))).round().astype(int)]
    vals, walls = [], []
    for step in range(args.warmup + args.steps):
        t = 0.0
        a = time.perf_counter()
        for sy in pick:
            cb = cpu_baseline(sy, args.cpu_budget)
            t += sy.n_basis / cb["value"]
        if step >= args.warmup:
            vals.append(sum(s.n_basis for s in systems) / (t * len(systems) / len(pick)))
            walls.append(time.perf_counter() - a)
    val = statistics.median(vals)
    ksum = sum(s.n_basis for s in systems)
    print(json.dumps({"impl": "reference", "metric": METRIC, "value": val, "unit": "P-columns/s",
                      "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
                      "ms_per_step": 1000.0 * statistics.median(walls),
                      "projected_ms_per_scf_step": 1000.0 * ksum / val,
                      "value_kind": "projected from a bounded sample per step",
                      "higher_is_better": True, "scaling": "weak",
                      "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                      "config": {"workload": args.workload, "systems": len(systems), "sum_n_basis": ksum},
                      "cpu_baseline": {"kind": "oracle", "cores": os.cpu_count(), "value": val, "unit": "P-columns/s",
                                       "sample": f"bounded one-step samples of {len(pick)} of {len(systems)} systems, "
                                                 "scaled by the system count"},
                      "e2e": {"value": val, "unit": "P-columns/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}),
          flush=True)


def run_reference(args, sysm, rank, world):
    if rank != 0:
        return
    res = []
    for i in range(args.warmup + args.steps):
        cb = cpu_baseline(sysm, args.cpu_budget)
        if i >= args.warmup:
            res.append(cb)
    val = statistics.median(r["value"] for r in res)
    # a step of this arm is one bounded sample: ms_per_step is the wall time it
    # took; value is the P-columns/s of a whole oracle SCF step projected from
    # it (projected_ms_per_scf_step)
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": "P-columns/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1000.0 * statistics.median(r["seconds"] for r in res),
            "projected_ms_per_scf_step": 1000.0 * sysm.n_basis / val,
            "value_kind": "projected from a bounded sample per step",
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": sysm.name, "n_basis": sysm.n_basis,
                                            "n_atoms": sysm.n_atoms, "grid": [int(x) for x in sysm.grid_n]},
            "cpu_baseline": {"kind": "oracle", "cores": res[0]["cores"], "sample": res[0]["sample"], "value": val,
                             "unit": "P-columns/s"},
            "e2e": {"value": val, "unit": "P-columns/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def expansion_roofline(infos, K, fp64, peak, peak_source):
    """Roofline of the Chebyshev expansion (moments and weighted sum): a
    polynomial of N_C terms and its moments take at least 2 sqrt(2 N_C)
    products of symmetric K x K matrices (the fewest products any grouping of
    s + 2 N_C / s needs), each K^2 (K + 1) flop, three times that in split 16-bit form; over the time of
    both passes, so that everything else in them counts as loss."""
    per = (1.0 if fp64 else 3.0) * K * K * (K + 1.0)
    rate = statistics.median(2.0 * (2.0 * i.n_cheb) ** 0.5 * per / ((i.ms_stage[3] + i.ms_stage[4]) / 1000.0)
                             for i in infos if i.ms_stage[3] + i.ms_stage[4] > 0) / 1e12
    return {"kernel": "k_ps_prod" if fp64 else "k_pst_prod", "bound": "alu" if fp64 else "tensor", "achieved": rate,
            "peak": peak, "unit": "TFLOP/s", "frac": rate / peak, "traffic": None, "peak_source": peak_source}


def tensor_peak(pk):
    return pk.get("bf16_tflops_sustained", 1700.0), (
        "MEASURED_PEAKS bf16_tflops_sustained (of measured; fp16 dense rate equals bf16)"
        if "bf16_tflops_sustained" in pk else "fallback 1700 TFLOP/s sustained (MEASURED_PEAKS.json absent)")


def max_over_ranks(value, world, device):
    """The largest of the ranks' values: the job is as slow as its slowest rank."""
    if world <= 1:
        return float(value)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(world, units_per_rank, steps, max_ms):
    """Units all ranks processed per second (weak scaling: every rank runs the
    same workload), timed by the slowest rank."""
    return world * units_per_rank * steps / (max_ms / 1000.0)


def main():
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    import workloads as w
    if args.workload.startswith("batch"):
        if args.impl == "reference":
            run_reference_batch(args, rank)
            return
        run_batched(args, rank, world)
        return
    sysm = w.config_system(args.workload)
    if args.impl == "reference":
        run_reference(args, sysm, rank, world)
        return
    import torch
    import torch.distributed as dist
    import paper_2108_13478_gb300 as dft
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl")
    prec = {"fp64": dft.DFT_PREC_FP64, "fp16x3": dft.DFT_PREC_FP16X3, "bf16x3": dft.DFT_PREC_BF16X3}[args.precision]
    stream = torch.cuda.current_stream()
    if args.time_to_solution:
        if rank == 0:
            rec = time_to_solution(args, dft, torch, local)
            print(json.dumps({"metric": "SCF wall time to the oracle's converged energy (<=1e-5 Ha/atom)",
                              "unit": "s", "higher_is_better": False, "data": "synthetic", **rec}), flush=True)
        return
    if args.dm_only:
        run_dm_only(args, dft, torch, sysm, prec, local, rank)
        return
    mixer = {"linear": dft.DFT_MIX_LINEAR, "kerker": dft.DFT_MIX_KERKER, "pulay": dft.DFT_MIX_PULAY}[args.mixer]
    reuse = 0 if (args.no_reuse_mu or prec == dft.DFT_PREC_FP64) else 1
    ctx = dft.Context(sysm, device=f"cuda:{local}", precision=prec, cheb_tail_tol=cheb_tail(args), mix_alpha=0.3,
                      mixer=mixer, kerker_q0=0.8, mix_history=8, reuse_mu=reuse,
                      model=dft.DFT_MODEL_NEUTRAL if args.model == "neutral" else dft.DFT_MODEL_LITERAL)
    ctx.overlap_kinetic()
    n = ctx.initial_density()
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device=f"cuda:{local}")

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
    for _ in range(args.warmup):
        ctx.scf_step(n)
    n_start = n.clone()          # the e2e leg re-runs the same SCF steps from here
    e_prev_state = None
    barrier()
    sampler = ClockSampler(local)
    sampler.start()
    launches0 = dft.dft_kernel_launches()
    step_ms, infos = [], []
    for _ in range(args.steps):
        flush.zero_()                      # L2 flush between timed steps (outside the events)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        info = ctx.scf_step(n)
        e1.record(stream)
        e1.synchronize()
        step_ms.append(e0.elapsed_time(e1))
        infos.append(info)
    barrier()
    launches = (dft.dft_kernel_launches() - launches0) / args.steps
    clocks = sampler.stop()
    total_ms = max_over_ranks(sum(step_ms), world, f"cuda:{local}")
    K = ctx.K
    value = job_throughput(world, K, args.steps, total_ms)
    # end to end through the public API with host buffers: pinned n_in -> device,
    # step, next density and energies back to the host
    n_host = torch.empty(ctx.grid_shape, dtype=torch.float64, pin_memory=True)
    n_host.copy_(n_start.cpu())
    out_host = torch.empty_like(n_host).pin_memory()
    dev_n = ctx.grid_array()
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e2e_ms = 0.0
    for _ in range(args.steps):
        flush.zero_()
        e0.record(stream)
        dev_n.copy_(n_host, non_blocking=True)
        info = ctx.scf_step(dev_n)
        out_host.copy_(dev_n, non_blocking=True)
        e1.record(stream)
        e1.synchronize()
        e2e_ms += e0.elapsed_time(e1)
        n_host.copy_(out_host)
    e2e_value = job_throughput(world, K, args.steps, max_over_ranks(e2e_ms, world, f"cuda:{local}"))
    pk = peaks()
    n_c = infos[-1].n_cheb
    sm_mhz = clocks.get("sm_mhz") or pk.get("sm_max_mhz", 2070.0)
    fp64 = prec == dft.DFT_PREC_FP64
    if fp64:
        roof = expansion_roofline(infos, K, True, FP64_FLOP_PER_SM_CLK * N_SM * sm_mhz * 1e6 / 1e12,
                                  "FP64 issue rate 4 flop/SM/clk x 152 SMs x median SM clock")
    else:
        roof = expansion_roofline(infos, K, False, *tensor_peak(pk))
    dtype = "f64" if fp64 else args.precision
    line = {"metric": METRIC, "value": value, "unit": "P-columns/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": dtype, "data": "synthetic",
            "config": {"workload": sysm.name, "n_basis": K, "n_atoms": sysm.n_atoms,
                       "grid": [int(x) for x in sysm.grid_n], "kT": sysm.kT, "n_cheb": n_c,
                       "cheb_tail_tol": cheb_tail(args), "model": args.model,
                       "mixer": args.mixer + " alpha 0.3" + (" kerker q0 0.8 hist 8" if args.mixer == "pulay" else ""),
                       "precision": args.precision, "l2": "flushed (256 MB write) between timed steps",
                       "parallelism": f"replicas x{world}"},
            "e2e": {"value": e2e_value, "unit": "P-columns/s",
                    "h2d_bytes_per_step": int(n_host.numel() * 8), "d2h_bytes_per_step": int(n_host.numel() * 8)},
            "gpu_launches": int(launches), "clocks": clocks, "roofline": roof,
            "stages_ms": [round(x, 3) for x in infos[-1].ms_stage],
            "stages_ms_median": [round(statistics.median(i.ms_stage[k] for i in infos), 3) for k in range(8)],
            "mu_reused_steps": int(sum(i.mu_reused for i in infos)),
            "energy_per_atom": infos[-1].e_total / sysm.n_atoms}
    if rank == 0 and not args.no_compare:
        line["mixed_vs_fp64"] = compare_precisions(dft, torch, local, cheb_tail(args))
    if rank == 0 and not args.no_sparse:
        line["sparse_route"] = sparse_route(dft, torch, local, cheb_tail(args), sm_mhz)
    if rank == 0 and prec != dft.DFT_PREC_FP64 and args.accuracy_workload != "none":
        del flush
        torch.cuda.empty_cache()
        line["dm_accuracy"] = dm_accuracy(dft, torch, local, args.accuracy_workload, cheb_tail(args))
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = {k: v for k, v in cpu_baseline(sysm, args.cpu_budget).items()
                                if k in ("value", "unit", "cores", "kind", "sample")}
    if rank == 0:
        print(json.dumps(line), flush=True)
    ctx.close()
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
