#!/usr/bin/env python
"""Benchmark: Cahn-Hilliard time steps per second at a 1e-8 true relative residual.

Workload (the 2D FP64 configuration): unit square split into 512 x 512 cells of two P1
triangles (263,169 nodes, 1,052,676 unknowns over the 4 fields), phi_p = phi_nfa = 0.33 +/- 0.01
(seeded SplitMix64 noise, seed 0), tau = 1e-4, eps = 1e-3, flux boundary conditions of the paper.
One step = loads + right-hand sides + FGMRES(30) with Algorithm 1 (smoothed-aggregation AMG
V-cycles) for both species to ||b - A x|| <= 1e-8 ||b|| + state update.

Prints one JSON line (rank 0).  `--impl reference` times the CPU oracle (direct solve) instead.
Under torchrun every rank runs an independent replica (the solve of one mesh does not shard).
"""
import os

for _v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")  # the oracle baseline runs on one core

import argparse
import json
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "CH time steps/s at 1e-8 rel. residual (FP64 vs mixed+learned); SpMV/AMG HBM %"
UNIT = "steps/s"
WORKLOAD_STEPS = 100  # the configuration's run length, used to amortise one-off set-up costs
FP64_FMA_PER_CLK_SM = 2  # GB300: 1.25 TFLOP/s FP64 nominal = 152 SMs x 2 FMA x 2 x 2.07 GHz
LEARNED_STEPS = 40  # timed steps per form in the learned warm-start section


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--nx", type=int, default=512)
    ap.add_argument("--ny", type=int, default=512)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-mixed", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-learned", action="store_true")
    ap.add_argument("--no-extra", action="store_true", help="skip the C1, mesh-size and 3D sections")
    ap.add_argument("--prewarm-s", type=float, default=2.0,
                    help="seconds of untimed steps on a throwaway state before the timed state exists")
    ap.add_argument("--learned-nx", type=int, default=256)
    return ap.parse_args()


def workload_name(nx, ny):
    n = (nx + 1) * (ny + 1)
    return (f"2D unit square {nx}x{ny} cells x 2 P1 triangles ({n} nodes, {4 * n} unknowns), "
            f"phi_p=phi_nfa=0.33+/-0.01 seed 0, tau=1e-4, eps=1e-3, flux BCs; FGMRES(30) + "
            f"Algorithm 1 (SA-AMG V-cycles) to 1e-8 true relative residual, both species")


# ---------------------------------------------------------------- oracle (CPU) timing
def oracle_rate(nx, ny, steps, warmup=0, keep=False):
    """Oracle steps/s on the same workload: assembly + LU once, amortised over the run length;
    `warmup` untimed steps run between the factorisation and the timed steps.  With keep, also
    returns the oracle's state after every step (warm-up steps included)."""
    import numpy as np
    from oracle import ch_oracle as o
    from paper_2204_03575_gb300 import inputs
    t0 = time.perf_counter()
    s = o.Solver(o.Params(nx=nx, ny=ny))
    t_setup = time.perf_counter() - t0
    pp, pn = inputs.initial_state(s.N, 0.33, 0.33, 0.01, seed=0)
    st = o.initial(s.N, pp, pn)
    states = []
    for _ in range(warmup):
        st = s.step(st)
        states.append(st)
    t0 = time.perf_counter()
    for _ in range(steps):
        st = s.step(st)
        if keep:
            states.append(st)
    t_steps = (time.perf_counter() - t0) / steps
    per_step = t_steps + t_setup / WORKLOAD_STEPS
    assert np.isfinite(st.phi_p).all()
    sample = (f"{nx}x{ny} oracle (numpy/scipy, SuperLU direct solve) on 1 of {os.cpu_count()} host cores: "
              f"assembly+factorisation {t_setup:.1f} s once, {warmup} untimed and {steps} timed steps at "
              f"{t_steps:.2f} s/step; rate = 1/(step + setup/{WORKLOAD_STEPS})")
    if keep:
        return 1.0 / per_step, sample, t_setup, t_steps, states
    return 1.0 / per_step, sample, t_setup, t_steps


def error_vs_oracle(gpu_traj, oracle_states):
    """Max over the four fields of ||x_gpu - x_oracle||_inf / ||x_oracle||_inf after each step of
    two runs from the same seeded initial state."""
    out = []
    for g, r in zip(gpu_traj, oracle_states):
        out.append(max(float(abs(g[k] - getattr(r, k)).max() / abs(getattr(r, k)).max())
                       for k in ("phi_p", "phi_nfa", "mu_p", "mu_nfa")))
    return out


def reference_main(args, rank):
    if rank != 0:
        return
    K = max(1, min(args.steps, 10))  # each oracle step takes seconds: a bounded sample
    W = max(0, min(args.warmup, 5))
    rate, sample, _, t_step = oracle_rate(args.nx, args.ny, K, warmup=W)
    line = {"impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
            "steps": K, "warmup": W, "ms_per_step": 1e3 / rate, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": workload_name(args.nx, args.ny), "parallelism": "rank 0 only"},
            "cpu_baseline": {"kind": "oracle", "value": rate, "unit": UNIT, "cores": 1,
                             "host_cores": os.cpu_count(),
                             "sample": sample + "; steps capped at 10, warm-up at 5"},
            "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------- clocks
class Clocks:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, dev):
        self.dev = dev
        self.p = None

    def __enter__(self):
        # The sampler's start-up (driver / NVML initialisation) must not overlap the timed region:
        # wait, up to 15 s, for its first sample before returning.
        import threading
        self.lines = []
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                       "-lms", "200", "-i", str(self.dev)], stdout=subprocess.PIPE,
                                      stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.p = None
            return self
        first = threading.Event()

        def read():
            for line in self.p.stdout:
                self.lines.append(line)
                first.set()
            first.set()

        self.reader = threading.Thread(target=read, daemon=True)
        self.reader.start()
        first.wait(timeout=15.0)
        self.skip = len(self.lines)  # samples taken before the timed region are not kept
        return self

    def __exit__(self, *a):
        self.out = ""
        if self.p is not None:
            self.p.terminate()
            try:
                self.p.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.p.kill()
                self.p.wait()
            self.reader.join(timeout=5)
            self.out = "".join(self.lines[self.skip:])

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in (self.out or "").splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ---------------------------------------------------------------- GPU timing
def make_solver(ch, nx, ny, precision):
    p = ch.Params(nx=nx, ny=ny, precision=precision)
    mesh = ch.Mesh(p)
    system = ch.System(mesh, p)
    pc = ch.Precond(system)
    state = ch.State(system, pc)
    state.init_seeded(0.33, 0.33, 0.01, seed=0)
    return system, pc, state


class Ranks:
    """The job's ranks (one process per GPU, replicas of the workload): a barrier around every timed
    region and the slowest rank's time, which is the whole job's time.  `device` holds the
    reduction tensor (cuda under NCCL, cpu under gloo)."""

    def __init__(self, world=1, dist=None, device="cpu"):
        self.world, self.dist, self.device = world, dist, device

    def barrier(self):
        if self.world > 1:
            self.dist.barrier()

    def max(self, ms):
        import torch
        t = torch.tensor([float(ms)], dtype=torch.float64, device=self.device)
        if self.world > 1:
            self.dist.all_reduce(t, op=self.dist.ReduceOp.MAX)
        return float(t.item())

    def rate(self, units_per_rank, ms_max):
        """Whole-job units per second: every rank did units_per_rank in at most ms_max."""
        return self.world * units_per_rank / (ms_max * 1e-3)


def timed_steps(torch, ch, state, K, flush, ranks, net=None):
    """K steps timed with CUDA events (ch_step, or ch_step_learned with `net`); returns the
    slowest rank's milliseconds and this rank's iteration counts."""
    iters = []
    torch.cuda.synchronize()
    ranks.barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(K):
        flush.zero_()  # 256 MiB write: evicts L2 between steps
        st = state.step() if net is None else state.step_learned(net)
        if st["status"] != 0 or max(st["relres"]) > 1e-8:
            raise RuntimeError(f"step did not reach 1e-8: {st}")
        iters.append(st["iters"])
    e1.record()
    torch.cuda.synchronize()
    ranks.barrier()
    return ranks.max(e0.elapsed_time(e1)), iters


def extra_sections(torch, ch, np, K, W, flush, ranks):
    """32x32 steps/s (10 steps), FGMRES iterations per step for 32^2 .. 512^2 (first 10 steps of
    the same seeded run), and 3D 128x128x32 Kuhn tetrahedra on [0,1]^2 x [0,0.25], bases
    0.30/0.30 +/- 0.01 seed 0, FP32 V-cycles in FP64 FGMRES, up to 50 timed steps."""
    out = {}
    _, _, st1 = make_solver(ch, 32, 32, precision=0)
    for _ in range(W):
        st1.step()
    ms1, it1 = timed_steps(torch, ch, st1, 10, flush, ranks)
    out["2d_32x32_fp64"] = {"steps": 10, "steps_per_s": ranks.rate(10, ms1),
                            "iters_per_step_mean": float(np.mean(it1)),
                            "note": "launch-bound: a roofline is not meaningful at 1089 nodes"}
    del st1
    scaling = {}
    for n in (32, 64, 128, 256, 512):
        _, pcn, stn = make_solver(ch, n, n, precision=0)
        its = [max(stn.step()["iters"]) for _ in range(10)]
        scaling[f"{n}x{n}"] = {"iters_per_step_mean_first10": float(np.mean(its)),
                               "amg_levels_H": [r for r, _ in pcn.levels(1)]}
        del pcn, stn
    out["fp64_iters_vs_mesh"] = scaling
    p3 = ch.Params(dim=3, nx=128, ny=128, nz=32, Lz=0.25, precision=1)
    sys3 = ch.System(ch.Mesh(p3), p3)
    pc3 = ch.Precond(sys3)
    st3 = ch.State(sys3, pc3)
    st3.init_seeded(0.30, 0.30, 0.01, seed=0)
    for _ in range(W):
        st3.step()
    K3 = min(K, 50)
    ms3, it3 = timed_steps(torch, ch, st3, K3, flush, ranks)
    ch.profile_enable(True)
    ch.profile_read(reset=True)
    for _ in range(5):
        flush.zero_()
        st3.step()
    torch.cuda.synchronize()
    prof3 = ch.profile_read(reset=True)
    ch.profile_enable(False)
    out["3d_128x128x32_mixed"] = {
        "workload": "3D [0,1]^2 x [0,0.25], 128x128x32 hexes x 6 Kuhn tetrahedra, phi_p=phi_nfa=0.30+/-0.01 "
                    "seed 0, FP32 V-cycles in FP64 FGMRES to 1e-8", "nodes": sys3.n, "nnz": sys3.nnz,
        "steps": K3, "steps_per_s": ranks.rate(K3, ms3), "ms_per_step": ms3 / K3,
        "iters_per_step_mean": float(np.mean(it3)), "amg_levels": {"M": [r for r, _ in pc3.levels(0)],
                                                                    "H": [r for r, _ in pc3.levels(1)]},
        "top_kernels": top_kernels(prof3)}
    del st3, pc3, sys3
    out["paper_minres"] = paper_section(torch, ch, flush, ranks)
    return out


def minres_case(torch, ch, flush, ranks, **kw):
    """One of the paper's solver experiments (Section 4): phi_p = phi_nfa = 0.35 +/- 0.01 (seed 0),
    preconditioned MINRES (krylov = 1; Algorithm 1 with fixed FP64 V-cycles) to a 1e-7 relative
    residual.  Iterations: the worse species of each of the first 20 steps (the figures' measure);
    time: the next 10 steps (CUDA events, L2 flushed between steps)."""
    p = ch.Params(krylov=1, rtol=1e-7, **kw)
    system = ch.System(ch.Mesh(p), p)
    state = ch.State(system, ch.Precond(system))
    state.init_seeded(0.35, 0.35, 0.01, seed=0)
    its = [max(state.step()["iters"]) for _ in range(20)]
    torch.cuda.synchronize()
    ranks.barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    worst, failed = 0.0, 0
    for _ in range(10):
        flush.zero_()
        st = state.step()
        failed += st["status"] != 0
        worst = max(worst, max(st["relres"]))
    e1.record()
    torch.cuda.synchronize()
    ranks.barrier()
    ms = ranks.max(e0.elapsed_time(e1)) / 10
    out = {"points": system.n, "minres_iters_max_first20": int(max(its)),
           "minres_iters_min_first20": int(min(its)), "minres_iters_first20": [int(i) for i in its],
           "ms_per_step_both_species": ms, "steps_per_s": ranks.rate(10, 10 * ms),
           "max_relres_timed": worst, "failed_steps_timed": int(failed)}
    del state, system
    return out


def paper_section(torch, ch, flush, ranks):
    """The paper's solver experiments on its boxes (Section 4): 2D 10 x 2.5 with nx x ny grid
    points (Fig. 1), 3D 10 x 2.5 x 10 with nx x ny x nz points (Fig. 3), and at 800 x 400 points
    the interface parameter (Fig. 4) and time step (Fig. 5) sweeps and the patterned substrate.
    tau 1e-4 and eps 1e-3 unless swept.  A case that raises is recorded, not fatal."""
    box2 = dict(Lx=10.0, Ly=2.5)
    box3 = dict(dim=3, Lx=10.0, Ly=2.5, Lz=10.0)
    groups = {
        "fig1_2d": {f"{a}x{b}": dict(nx=a - 1, ny=b - 1, **box2)
                    for a, b in ((100, 50), (200, 100), (400, 200), (800, 400), (1600, 800))},
        "fig3_3d": {f"{a}x{b}x{c}": dict(nx=a - 1, ny=b - 1, nz=c - 1, **box3)
                    for a, b, c in ((30, 15, 30), (40, 20, 40), (60, 30, 60), (80, 40, 80),
                                    (120, 60, 120), (160, 80, 160))},
        "fig4_eps_800x400": {f"eps={e:g}": dict(nx=799, ny=399, eps=e, **box2) for e in (1e-2, 1e-1, 1.0, 10.0)},
        "fig5_tau_800x400": {f"tau={t:g}": dict(nx=799, ny=399, tau=t, **box2) for t in (1e-7, 1e-6, 1e-5)},
        "patterned_800x400": {"pattern=1": dict(nx=799, ny=399, pattern=1, **box2)},
    }
    out = {}
    for g, cases in groups.items():
        out[g] = {}
        for name, kw in cases.items():
            try:
                out[g][name] = minres_case(torch, ch, flush, ranks, **kw)
            except ch.ChError as e:  # a library status (e.g. out of memory) raised by the binding
                out[g][name] = {"error": str(e)[:200]}
    return out


def variants_section(torch, ch, np, nx, K, W, flush, ranks):
    """The solver's variants on the headline workload (nx x nx, seeded 0.33 +/- 0.01): M~ by the
    Chebyshev semi-iteration (precond_M = 1, Section 3) in FP64 and mixed precision, and the
    Flory-Huggins potential (potential = 3, Section 2) in FP64; K timed steps after W warm-up
    steps each, every step at the true 1e-8 residual."""
    out = {}
    for tag, kw in (("chebyshev_M_fp64", dict(precond_M=1)), ("chebyshev_M_mixed", dict(precond_M=1, precision=1)),
                    ("flory_huggins_fp64", dict(potential=3))):
        p = ch.Params(nx=nx, ny=nx, **kw)
        system = ch.System(ch.Mesh(p), p)
        state = ch.State(system, ch.Precond(system))
        state.init_seeded(0.33, 0.33, 0.01, seed=0)
        for _ in range(W):
            state.step()
        ms, iters = timed_steps(torch, ch, state, K, flush, ranks)
        out[tag] = {"steps": K, "steps_per_s": ranks.rate(K, ms), "ms_per_step": ms / K,
                    "iters_per_step_mean": float(np.mean(iters)), "params": {k: int(v) for k, v in kw.items()}}
        del state, system
    return out


def eoc_section(torch, ch, np):
    """Section 4's convergence study in tau: five step sizes 2e-4 .. 3.2e-3 against tau = 1e-5 on
    the paper's 10 x 2.5 box, 0.35 +/- 0.01 (seed 0), eps = 1e-3, Eq. (15), final time T = 3.2e-2
    (ten steps of the largest tau; 3200 of the reference); FP64 solves to a 1e-10 residual.  The
    paper states neither the mesh nor T nor the norm: two grids are run, its smallest 2D grid
    (100 x 50 points) and a coarse 16 x 8.  Errors in the discrete L2 norm sqrt(e^T M e); a run
    whose state leaves [-10, 10] has diverged (the explicit potential term blows up at large tau
    on fine meshes) and is left out of the orders, which are pairwise (successive tau) and a
    least-squares fit of log(error) on log(tau) over the stable runs."""
    import math
    import scipy.sparse as sp
    T, taus = 3.2e-2, (2e-4, 4e-4, 8e-4, 1.6e-3, 3.2e-3)
    out = {"final_time": T, "reference_tau": 1e-5, "taus": list(taus), "box": "10 x 2.5",
           "paper_eoc": {"polymer": 0.789, "nfa": 0.788}}
    t0 = time.time()
    for nx, ny in ((99, 49), (15, 7)):
        def run(tau):
            p = ch.Params(nx=nx, ny=ny, Lx=10.0, Ly=2.5, tau=tau, rtol=1e-10)
            system = ch.System(ch.Mesh(p), p)
            state = ch.State(system, ch.Precond(system))
            state.init_seeded(0.35, 0.35, 0.01, seed=0)
            n = int(round(T / tau))
            ok = True
            for _ in range(n):
                st = state.step(check=False)
                if st["status"] != 0:
                    ok = False
                    break
            g = state.get()
            pp, pn = g["phi_p"].cpu().numpy(), g["phi_nfa"].cpu().numpy()
            ok = ok and bool(np.isfinite(pp).all() and np.abs(pp).max() < 10 and np.abs(pn).max() < 10)
            return pp, pn, system, n, ok

        rp, rn, system, nref, _ = run(1e-5)
        rowptr, col, vm, _, _ = [t.cpu().numpy() for t in system.csr()]
        M = sp.csr_matrix((vm, col, rowptr), shape=(system.n, system.n))

        def mnorm(d):
            return math.sqrt(float(d @ (M @ d)))

        errs, stable = {"polymer": [], "nfa": []}, []
        for tau in taus:
            pp, pn, _, _, ok = run(tau)
            stable.append(ok)
            errs["polymer"].append(mnorm(pp - rp) if ok else None)
            errs["nfa"].append(mnorm(pn - rn) if ok else None)
        g = {"grid_points": f"{nx + 1} x {ny + 1}", "reference_steps": nref, "stable": stable}
        keep = [i for i, ok in enumerate(stable) if ok]
        for k, e in errs.items():
            ek = np.array([e[i] for i in keep])
            tk = np.array([taus[i] for i in keep])
            g[k] = {"l2_error": e,
                    "eoc_pairwise": (np.log(ek[1:] / ek[:-1]) / np.log(tk[1:] / tk[:-1])).tolist() if len(ek) > 1 else [],
                    "eoc_fit": float(np.polyfit(np.log(tk), np.log(ek), 1)[0]) if len(ek) > 1 else None}
        out[f"{nx + 1}x{ny + 1}"] = g
    out["seconds"] = round(time.time() - t0, 1)
    return out


def morphology_section(torch, ch, state_fields, nx, reps=20):
    """Section 5's projection of the headline run's final morphology (nx x nx nodal image,
    polymer where phi_p > phi_nfa) onto the centres of a 2nx x 2nx finite-difference grid,
    upward ray-crossing parity per grid point; CUDA-event time over `reps` launches."""
    pp, pn = state_fields["phi_p"], state_fields["phi_nfa"]
    g = 2 * nx
    ch.morphology_project(pp, pn, nx, nx, 1.0, 1.0, g, g)  # warm-up
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        polymer, _, _ = ch.morphology_project(pp, pn, nx, nx, 1.0, 1.0, g, g)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / reps
    return {"image": f"{nx + 1} x {nx + 1}", "grid": f"{g} x {g}", "ms_per_projection": ms,
            "grid_points_per_s": g * g / (ms * 1e-3), "polymer_fraction": float(polymer.float().mean())}


def learned_section(torch, ch, nx, K, flush, ranks):
    """The learned warm start on an nx x nx grid: 2000 (s_{k-2}, s_{k-1}, s_k, s_{k+1}) quadruples
    from the plain FP64 solver (20 seeded runs x 100 steps), residual-loss training by the library's
    kernels, then K timed steps of a held-out run per form: previous-state guess, the network (a
    learned second-order extrapolation), linear extrapolation (the zero network) and quadratic
    extrapolation (theta = 1), in FP64 and mixed precision; plus the network's share of a learned
    step and its convolutions' tensor throughput."""
    import time
    import numpy as np
    from paper_2204_03575_gb300 import warmstart as ws
    t0 = time.time()
    data = ws.generate_pairs(nx, nx, seeds=range(20), steps=100, dtype=torch.float64)
    torch.cuda.synchronize()
    t_gen = time.time() - t0
    system = ws.make_system(nx, nx)
    net = ch.WarmStartNet(nx + 1, nx + 1, max_batch=8)
    t0 = time.time()
    net, info = ws.train_residual(data, net, system, epochs=8, batch=8, lr=2e-3)
    torch.cuda.synchronize()
    t_train = time.time() - t0
    del data
    zero, quad = ws.zero_net(nx, nx), ws.quadratic_net(nx, nx)
    out = {"workload": f"2D {nx}x{nx} P1 triangles ({(nx + 1) ** 2} nodes), held-out seed 1000, bases from "
                       f"SplitMix64 in [0.20, 0.45), noise +/-0.01; timed steps 4..{K + 3} of the run",
           "pairs": info["pairs"], "generate_s": round(t_gen, 2), "train_s": round(t_train, 2),
           "train_loss_first_last_epoch": [info["loss_per_epoch"][0], info["loss_per_epoch"][-1]],
           "held_out_loss_per_epoch": info["held_out_loss_per_epoch"],
           "held_out_loss_quadratic": info["held_out_loss_quadratic"], "selected": info["selected"],
           "selection": "fewest FGMRES iterations per step on a validation run (seed 999, steps 4..43) among "
                        "theta = 1, per-field constants (theta_phi, theta_mu) fitted on that run by a "
                        "coordinate search, and the network (started from those constants) after each epoch",
           "constant_theta": info["constant_theta"],
           "selection_iterations_quadratic_then_epochs": info["selection_scores_quadratic_then_epochs"],
           "loss_meaning": "mean ln(|r|^2 / |r_linear extrapolation|^2) of the step residual; the last 10% of "
                           "the pairs (2 of the 20 seeds) held out",
           "out_scale_theta_star": info["out_scale"]}
    forms = (("previous_state", None), ("learned", net), ("linear_extrapolation", zero),
             ("quadratic_extrapolation", quad))
    for prec, tag in ((0, "fp64"), (1, "mixed")):
        res = {}
        # one solver per precision: the forms share its hierarchy and autotuned launch shapes, so
        # they differ only in the initial guess; re-seeding restarts the run and the learned history
        state = ws.make_state(nx, nx, prec)
        # one prediction per network and one step from a guess before any timing: the first use of
        # the prediction's kernels in the process (module loading), each network's weight conversion
        # and the capture of the solver's guess-step graph stay out of the timed windows
        state.init_seeded(0.33, 0.33, 0.01, seed=0)
        state.step()
        s4 = state.state4()
        for _, n in forms:
            if n is not None:
                n.predict(s4, s4, s4)
        state.step_guess(s4)
        torch.cuda.synchronize()
        for form, n in forms:
            b0, b1 = ws.seed_bases(1000)
            state.init_seeded(b0, b1, 0.01, seed=1000)
            for _ in range(3):  # ch_step_learned starts from the previous state for three steps
                if n is None:
                    state.step()
                else:
                    state.step_learned(n)
            ms, iters = timed_steps(torch, ch, state, K, flush, ranks, net=n)
            res[form] = {"steps_per_s": ranks.rate(K, ms), "ms_per_step": ms / K,
                         "iters_per_step_mean": float(np.mean(iters))}
        if prec == 0:  # the network's share of a learned step (per-launch event timing)
            b0, b1 = ws.seed_bases(1000)
            state.init_seeded(b0, b1, 0.01, seed=1000)
            for _ in range(3):
                state.step_learned(net)
            ch.profile_enable(True)
            ch.profile_read(reset=True)
            for _ in range(5):
                flush.zero_()
                state.step_learned(net)
            torch.cuda.synchronize()
            prof = ch.profile_read(reset=True)
            ch.profile_enable(False)
            tot = sum(v["ms"] for v in prof.values()) or 1.0
            conv = prof.get("ws_conv_f32", {"ms": 0.0, "fmas": 0.0, "launches": 0})
            io = prof.get("ws_io_f64", {"ms": 0.0})
            out["network_share_of_learned_step"] = (conv["ms"] + io["ms"]) / tot
            out["conv_tflops"] = (2 * conv["fmas"] / (conv["ms"] * 1e-3) / 1e12) if conv["ms"] > 0 else None
            out["conv_ms_per_prediction"] = conv["ms"] / 5
        out[tag] = res
    out["mixed_learned_over_fp64_previous_state"] = (out["mixed"]["learned"]["steps_per_s"]
                                                     / out["fp64"]["previous_state"]["steps_per_s"])
    return out


def roofline(prof, peaks, seq=None):
    """Dominant kernel (largest summed event time) against its bound.  Both fractions are given:
    frac_hbm (algorithmic bytes per launch / launch time against the measured HBM copy rate: the
    unit of the >= 60 % target for SpMV and V-cycle kernels) and, for FP64 kernels, frac_alu
    (FMAs against the FP64 pipe's peak).  `bound`/`frac` name the one that binds the kernel.
    With `seq` (the kernel timed as the solve runs it: back-to-back launches in one CUDA graph,
    `smoother_in_sequence`) the launch time is that one; the per-launch event timing, which
    isolates every launch between two events, is kept under `event_timed`."""
    name, e = max(prof.items(), key=lambda kv: kv[1]["ms"])
    if name not in ("cheb_step_f64", "cheb_step_f32"):
        seq = None  # the in-sequence timing is of the fine-level Chebyshev step only
    hbm = peaks.get("hbm_gbs", 6800.0)
    fp64_peak = 152 * FP64_FMA_PER_CLK_SM * 2 * peaks.get("sm_max_mhz", 2070.0) * 1e6 / 1e12  # TFLOP/s
    fmas_per_byte = e["fmas"] / max(e["bytes"], 1.0)
    alu_balance = fp64_peak * 1e12 / 2 / (hbm * 1e9)  # FP64 FMA per byte at which both bounds meet
    bytes_pl, fmas_pl = e["bytes"] / e["launches"], e["fmas"] / e["launches"]

    def rates(us):
        r = {"avg_launch_us": us, "achieved_GBps": bytes_pl / (us * 1e-6) / 1e9}
        r["frac_hbm"] = r["achieved_GBps"] / hbm
        if name.endswith("f64"):
            r["achieved_TFLOPs_fp64"] = 2 * fmas_pl / (us * 1e-6) / 1e12
            r["frac_alu"] = r["achieved_TFLOPs_fp64"] / fp64_peak
        return r

    ev = rates(1e3 * e["ms"] / e["launches"])
    out = {"kernel": name, "launches": e["launches"],
           "share_of_kernel_time": e["ms"] / sum(v["ms"] for v in prof.values())}
    main = rates(seq["avg_launch_us"]) if seq else ev
    out.update(main)
    out["timing"] = ("in sequence: back-to-back launches of the kernel in one CUDA graph, as the solve runs "
                     "them (in_sequence); event_timed: CUDA events around each launch of 20 bench steps"
                     if seq else "CUDA events around each launch of 20 bench steps")
    if seq:
        out["event_timed"] = ev
        out["in_sequence"] = seq
    hbm_src = "measured (MEASURED_PEAKS.json hbm_gbs)" if "hbm_gbs" in peaks else "fallback"
    if name.endswith("f64") and fmas_per_byte > alu_balance:
        out.update({"bound": "alu", "achieved": main["achieved_TFLOPs_fp64"], "peak": fp64_peak,
                    "unit": "TFLOP/s", "frac": main["frac_alu"],
                    "peak_source": "derived: 152 SMs x 2 FP64 FMA/clk x 2 flops x max SM clock "
                                   "(measured probe: 1.20 TFLOP/s); frac_hbm against " + hbm_src})
    else:
        out.update({"bound": "hbm", "achieved": main["achieved_GBps"], "peak": hbm, "unit": "GB/s",
                    "frac": main["frac_hbm"], "peak_source": hbm_src})
        if main["frac_hbm"] > 1.0:
            out["note"] = ("the kernel's working set at this size stays in the 129 MB L2 between launches, so "
                           "it runs above the HBM rate; fine_smoother_hbm_bound times it where HBM binds")
    out["target"] = "frac_hbm >= 0.6 (HBM roofline of the SpMV / V-cycle kernels)"
    out["algorithmic_bytes_per_launch"] = bytes_pl
    out["fmas_per_launch"] = fmas_pl
    out["traffic"] = traffic_for(name)
    return out


def smoother_in_sequence(torch, ch, flush, pc, n, precision, passes=40, degree=5, reps=5):
    """The fine level's Chebyshev step timed as the solve runs it: ch_smooth (H's hierarchy,
    `passes` passes of `degree` steps, the solver's own kernels with its programmatic dependent
    launches) captured in one CUDA graph and replayed after an L2 flush; the time per launch is the
    graph's event time over its launches (the steps plus two vector loads and one store).
    Algorithmic bytes and FMAs are the library's own launch accounting of the same call."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(0)
    b = torch.randn(n, 2, dtype=torch.float64, device=dev, generator=g)
    x0 = torch.randn(n, 2, dtype=torch.float64, device=dev, generator=g)
    x = x0.clone()
    ch.profile_read(reset=True)
    pc.smooth(1, b, x, degree, passes)
    torch.cuda.synchronize()
    acc = ch.profile_read(reset=True)
    launches = sum(v["launches"] for v in acc.values())
    nbytes = sum(v["bytes"] for v in acc.values())
    fmas = sum(v["fmas"] for v in acc.values())
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(graph, stream=s):
            pc.smooth(1, b, x, degree, passes, stream=s)
    torch.cuda.current_stream().wait_stream(s)
    torch.cuda.synchronize()
    times = []
    for _ in range(reps):
        x.copy_(x0)
        flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        graph.replay()
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    ms = float(statistics.median(times))
    del graph
    return {"nodes": n, "precision": "fp32" if precision else "fp64", "launches": launches,
            "steps": passes * degree, "avg_launch_us": 1e3 * ms / launches,
            "bytes_per_launch": nbytes / launches, "achieved_GBps": nbytes / (ms * 1e-3) / 1e9,
            "achieved_TFLOPs": 2 * fmas / (ms * 1e-3) / 1e12,
            "how": f"ch_smooth (H, {passes} passes x degree {degree}) in one CUDA graph, L2 flushed "
                   f"before each of {reps} replays (median)"}


def in_sequence(torch, ch, flush, peaks, pc, n, precision, passes=40):
    """smoother_in_sequence with its fractions of the measured HBM rate and, in FP64, of the FP64
    pipe's peak."""
    r = smoother_in_sequence(torch, ch, flush, pc, n, precision, passes=passes)
    r["frac_hbm"] = r["achieved_GBps"] / peaks.get("hbm_gbs", 6800.0)
    if not precision:
        r["frac_alu"] = r["achieved_TFLOPs"] / (152 * FP64_FMA_PER_CLK_SM * 2 * peaks.get("sm_max_mhz", 2070.0)
                                                * 1e6 / 1e12)
    return r


def hbm_bound_smoother(torch, ch, flush, peaks):
    """The same kernel on a 2048 x 2048 lattice in FP32: its fine level (4.2 M rows, ~270 MB of
    operator and vectors) exceeds the 129 MB L2, so the steps stream from HBM."""
    p = ch.Params(nx=2048, ny=2048, precision=1)
    system = ch.System(ch.Mesh(p), p)
    pc = ch.Precond(system)
    r = in_sequence(torch, ch, flush, peaks, pc, system.n, 1, passes=20)
    r["workload"] = "2D 2048x2048 P1 lattice (4,198,401 nodes), H's finest level, FP32"
    del pc, system
    torch.cuda.synchronize()
    return r


def traffic_for(kernel):
    path = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    if not os.path.exists(path):
        return None
    try:
        d = json.load(open(path))
        return d.get(kernel, {}).get("bytes_per_launch")
    except (OSError, ValueError):
        return None


def top_kernels(prof, n=8):
    tot = sum(v["ms"] for v in prof.values()) or 1.0
    rows = sorted(prof.items(), key=lambda kv: -kv[1]["ms"])[:n]
    out = {}
    for k, v in rows:
        ms = v["ms"] / max(v["launches"], 1)
        out[k] = {"launches": v["launches"], "share": v["ms"] / tot,
                  "GBps": v["bytes"] / v["launches"] / (ms * 1e-3) / 1e9 if ms > 0 else None,
                  "GFMAps": v["fmas"] / v["launches"] / (ms * 1e-3) / 1e9 if ms > 0 else None}
    return out


# what the printed line keeps of the sections whose full form goes to stderr
SECTION_KEYS = {
    "roofline": ("kernel", "bound", "achieved", "peak", "unit", "frac", "peak_source", "share_of_kernel_time",
                 "avg_launch_us", "traffic"),
    "mixed": ("value", "ms_per_step", "iters_per_step_mean", "max_rel_diff_phi_vs_fp64_form_after_run"),
    "batch": ("runs", "nodes", "run_steps_per_s", "ms_per_step", "launches_per_step", "max_relres_last_step"),
    "cpu_baseline": ("value", "unit", "cores", "host_cores", "kind", "sample"),
    "learned": ("selected", "fp64", "mixed", "mixed_learned_over_fp64_previous_state"),
    "fine_smoother_hbm_bound": ("avg_launch_us", "achieved_GBps", "frac_hbm"),
}
DETAIL_ONLY = ("top_kernels", "configs", "variants", "eoc_tau", "morphology_projection")


def stdout_line(line):
    """The JSON line for stdout: the measurement and its context, 3 to 4 kB.  Readers that keep the tail of a run's
    output cut a line of 20 kB; the sections in full are on stderr ("bench detail: ")."""
    out = {k: v for k, v in line.items() if k not in DETAIL_ONLY}
    for name, keys in SECTION_KEYS.items():
        if isinstance(out.get(name), dict):
            out[name] = {k: out[name][k] for k in keys if k in out[name]}
    out["detail"] = "stderr"
    return out


def main():
    args = parse()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        reference_main(args, rank)
        return

    import numpy as np
    import torch
    import torch.distributed as dist
    from paper_2204_03575_gb300 import ch

    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    ranks = Ranks(world, dist, torch.device("cuda", local))
    barrier = ranks.barrier

    peaks = {}
    pk = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pk):
        peaks = json.load(open(pk))
    dev = torch.device("cuda", local)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    # the first zero_() loads PyTorch's fill kernel (lazy module loading: ~0.25 s on a fresh box);
    # do it before any timed region, which runs one flush per step
    flush.zero_()
    torch.cuda.synchronize()
    K, W = args.steps, max(args.warmup, 0)

    # ---- GPU pre-warm: an idle GPU ramps its clocks over the first fraction of a second; steps of
    # a throwaway solver of the same workload bring it to its working state before any timing
    if args.prewarm_s > 0:
        import time
        # autotune = 0: the throwaway solver leaves the per-process tuning cache empty, so the timed
        # solvers' SpMV widths are chosen on the warmed GPU
        pW = ch.Params(nx=args.nx, ny=args.ny, autotune=0)
        sysW = ch.System(ch.Mesh(pW), pW)
        pcW = ch.Precond(sysW)
        stateW = ch.State(sysW, pcW)
        stateW.init_seeded(0.33, 0.33, 0.01, seed=0)
        t0 = time.time()
        while time.time() - t0 < args.prewarm_s:
            stateW.step()
        torch.cuda.synchronize()
        del sysW, pcW, stateW

    # ---- FP64 form: the headline number
    system, pc, state = make_solver(ch, args.nx, args.ny, precision=0)
    N = system.n
    for _ in range(W):
        state.step()
    ch.profile_read(reset=True)
    with Clocks(local) as clk:
        ms, iters = timed_steps(torch, ch, state, K, flush, ranks)
    launches = sum(v["launches"] for v in ch.profile_read(reset=True).values())
    value = ranks.rate(K, ms)  # ms is already the slowest rank's
    fields64 = {k: v.clone() for k, v in state.get().items()}

    # ---- per-kernel event timing of the same steps (separate pass: events add host overhead)
    PK = min(K, 20)
    ch.profile_enable(True)
    ch.profile_read(reset=True)
    for _ in range(PK):
        flush.zero_()
        state.step()
    torch.cuda.synchronize()
    prof64 = ch.profile_read(reset=True)
    ch.profile_enable(False)
    roof = roofline(prof64, peaks, in_sequence(torch, ch, flush, peaks, pc, N, 0))

    # ---- end to end through the public API with host buffers
    sysE, pcE, stateE = make_solver(ch, args.nx, args.ny, precision=0)
    for _ in range(W):
        stateE.step()
    g = stateE.get()
    h_in = torch.stack([g["phi_p"], g["phi_nfa"]]).cpu().pin_memory()
    h_out = torch.empty((5, N), dtype=torch.float64).pin_memory()
    d_in = torch.empty((2, N), dtype=torch.float64, device=dev)
    mu = [g["mu_p"].clone(), g["mu_nfa"].clone()]
    torch.cuda.synchronize()
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(K):
        d_in.copy_(h_in, non_blocking=True)
        stateE.set(d_in[0], d_in[1], mu[0], mu[1])
        stateE.step()
        g = stateE.get()
        for i, k in enumerate(("phi_p", "phi_nfa", "phi_s", "mu_p", "mu_nfa")):
            h_out[i].copy_(g[k], non_blocking=True)
        mu = [g["mu_p"], g["mu_nfa"]]
        torch.cuda.current_stream().synchronize()
        h_in.copy_(h_out[0:2])
    e1.record()
    torch.cuda.synchronize()
    barrier()
    ms_e2e = ranks.max(e0.elapsed_time(e1))
    e2e = {"value": ranks.rate(K, ms_e2e), "unit": UNIT, "h2d_bytes_per_step": 2 * 8 * N,
           "d2h_bytes_per_step": 5 * 8 * N,
           "api": "ch_state_set / ch_step / ch_state_get with pinned host copies each step"}
    del sysE, pcE, stateE

    # ---- mixed precision form (FP32 AMG inside FP64 FGMRES)
    mixed = None
    if not args.no_mixed:
        sysM, pcM, stateM = make_solver(ch, args.nx, args.ny, precision=1)
        for _ in range(W):
            stateM.step()
        ms_m, iters_m = timed_steps(torch, ch, stateM, K, flush, ranks)
        fm = stateM.get()
        diff = max(float((fm[k] - fields64[k]).abs().max() / fields64[k].abs().max()) for k in ("phi_p", "phi_nfa"))
        ch.profile_enable(True)
        ch.profile_read(reset=True)
        for _ in range(PK):
            flush.zero_()
            stateM.step()
        torch.cuda.synchronize()
        profm = ch.profile_read(reset=True)
        ch.profile_enable(False)
        mixed = {"value": ranks.rate(K, ms_m), "ms_per_step": ms_m / K,
                 "iters_per_step_mean": float(np.mean(iters_m)),
                 "max_rel_diff_phi_vs_fp64_form_after_run": diff,
                 "roofline": roofline(profm, peaks, in_sequence(torch, ch, flush, peaks, pcM, N, 1)),
                 "top_kernels": top_kernels(profm)}
        del sysM, pcM, stateM

    # ---- batched workload: 64 independent runs of uneven size in one state (FP32 V-cycles)
    batch = None
    # the auxiliary sections below run at N = 1 only: N replicas would repeat them without adding
    # information while holding all N GPUs for minutes
    if not args.no_batch and world == 1:
        from paper_2204_03575_gb300 import inputs
        spec = inputs.batch_runs(64, seed=0)
        pb = ch.Params(precision=1)
        bmesh = ch.Mesh(pb, runs=[ch.Params(nx=nx, ny=ny) for nx, ny, _, _ in spec])
        bsys = ch.System(bmesh, pb)
        bstate = ch.State(bsys, ch.Precond(bsys))
        bstate.init_seeded_batch([x[2] for x in spec], [x[3] for x in spec], 0.01, seed=0)
        for _ in range(W):
            bstate.step()
        KB = min(K, 20)
        ch.profile_read(reset=True)
        ms_b, iters_b = timed_steps(torch, ch, bstate, KB, flush, ranks)
        blaunch = sum(v["launches"] for v in ch.profile_read(reset=True).values())
        worst = max(max(bstate.run_stats(r)["relres"]) for r in range(len(spec)))
        by_size = {}
        for r, (nx_r, ny_r, _, _) in enumerate(spec):
            by_size.setdefault(f"{nx_r}x{ny_r}", []).append(max(bstate.run_stats(r)["iters"]))
        per_size = {k: {"runs": len(v), "iters_last_step_mean": float(np.mean(v))} for k, v in sorted(by_size.items())}
        batch = {"workload": "64 runs, nx, ny drawn from {64,96,128,192,256}, bases U[0.20,0.45), "
                             "noise +/-0.01, FP32 V-cycles in FP64 FGMRES, one state (disjoint union)",
                 "runs": len(spec), "nodes": bsys.n, "steps": KB,
                 "run_steps_per_s": ranks.rate(len(spec) * KB, ms_b), "ms_per_step": ms_b / KB,
                 "launches_per_step": blaunch / KB, "max_relres_last_step": worst, "per_size": per_size}
        del bstate, bsys, bmesh

    # ---- the other configurations' throughput lines: 32x32 (launch-bound), FGMRES iterations per
    # step against the mesh size, and the 3D Kuhn-tetrahedra box in the mixed form
    extra = None
    if not args.no_extra and world == 1:
        extra = extra_sections(torch, ch, np, K, W, flush, ranks)

    # ---- the solver's variants (Chebyshev M~, Flory-Huggins), Section 4's EOC study in tau and
    # Section 5's morphology projection
    variants = eoc = morph = smoother_hbm = None
    if not args.no_extra and world == 1:
        variants = variants_section(torch, ch, np, args.nx, min(K, 20), W, flush, ranks)
        eoc = eoc_section(torch, ch, np)
        morph = morphology_section(torch, ch, fields64, args.nx)
        smoother_hbm = hbm_bound_smoother(torch, ch, flush, peaks)

    # ---- learned warm start (256 x 256 grid): training, then FP64 / mixed with and without it
    learned = None
    if not args.no_learned and world == 1:
        # a fixed window, steps 4..43 of the held-out run (the forms differ most in the first steps;
        # the window is the section's workload, not the headline's step count)
        learned = learned_section(torch, ch, args.learned_nx, LEARNED_STEPS, flush, ranks)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        # the GPU's FP64 and mixed trajectories of the first steps from the seeded state, at the
        # default 1e-8 tolerance, next to the oracle's (exact direct solves) of the same steps
        CB_W, CB_K = 1, 5
        traj = {}
        for prec, tag in ((0, "fp64"), (1, "mixed")):
            _, _, stT = make_solver(ch, args.nx, args.ny, precision=prec)
            t = []
            for _ in range(CB_W + CB_K):
                stT.step()
                t.append({k: v.cpu().numpy() for k, v in stT.get().items()})
            traj[tag] = t
            del stT
        rate, sample, _, _, ostates = oracle_rate(args.nx, args.ny, CB_K, warmup=CB_W, keep=True)
        cpu = {"value": rate, "unit": UNIT, "cores": 1, "host_cores": os.cpu_count(), "kind": "oracle",
               "sample": sample,
               "error_vs_oracle_per_step": {tag: error_vs_oracle(t, ostates) for tag, t in traj.items()},
               "error_note": "max over phi_p, phi_nfa, mu_p, mu_nfa of the relative inf-norm difference "
                             "between the GPU run (rtol 1e-8) and the oracle's run after each of the "
                             f"first {CB_W + CB_K} steps from the same seeded state"}

    levels = {"M": pc.levels(0), "H": pc.levels(1)}
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K, "warmup": W,
        "ms_per_step": ms / K, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_name(args.nx, args.ny), "nodes": N, "unknowns": 4 * N,
                   "l2": "flushed between steps (256 MiB write inside the timed region)",
                   "gpu_prewarm_s": args.prewarm_s,
                   "parallelism": "replicas" if world > 1 else "single GPU"},
        "clocks": clk.summary(), "e2e": e2e, "gpu_launches": launches, "launches_per_step": launches / K,
        "roofline": roof,
        "top_kernels": top_kernels(prof64),
        "iters_per_step_mean": float(np.mean(iters)), "iters_per_step_max": int(np.max(iters)),
        "amg_levels": {k: [r for r, _ in v] for k, v in levels.items()},
        "mixed": mixed, "batch": batch, "learned": learned, "configs": extra, "variants": variants,
        "eoc_tau": eoc, "morphology_projection": morph, "fine_smoother_hbm_bound": smoother_hbm,
        "cpu_baseline": cpu,
    }
    if rank == 0:
        print("bench detail: " + json.dumps(line), file=sys.stderr, flush=True)
        print(json.dumps(stdout_line(line)), flush=True)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
