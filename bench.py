#!/usr/bin/env python
"""Throughput of the forest-closeness hot path on GB300.

One step = the whole path on one batch: build G* from the CSR (validation,
degrees, start order, selector thresholds), sample tau = 1024 uniform spanning
trees of G* (Algorithm 2, one persistent launch), aggregate the u*-edge and
control-variate counts, Algorithm 1's pivot solve (CG on I + alpha L, FP32
inner / FP64 refinement to 1e-9), combination + farness + closeness (Eq. 3,
Def. 2) and the top-100 ranking.

Workload: Barabasi-Albert n = 2^20, m = 8 (seed clique K_9, seed 2),
unweighted, alpha = 1, tau = 1024 trees per step (synthetic stand-in for the
paper's complex networks).  Metric: USTs/s (trees per second, whole job).  The
default line also carries "time_to_eps": time to max-abs diag(Omega) error 0.1
on R-MAT scale 22 (edge factor 16, a = 0.57, b = c = 0.19), learned control
variate vs the plain estimator and the ablations (untrained network, g = p_v)
and the Rao-Blackwellised estimator, medians over 5 seeds.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun (N > 1) each rank samples its own 1024 trees of a N * 1024-tree
run (tree_offset = rank * 1024, weak scaling) and the ranks sum R and C with one
all-reduce before the combination; rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

N_LOG2, BA_M, BA_SEED, ALPHA, TAU, TOPK = 20, 8, 2, 1.0, 1024, 100
WORKLOAD = f"BA n=2^{N_LOG2} m={BA_M} (seed {BA_SEED}) unweighted, alpha={ALPHA:g}, tau={TAU} trees/step"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--tau", type=int, default=TAU)
    ap.add_argument("--n-log2", type=int, default=N_LOG2,
                    help="BA size 2^k (profiling cases only; the benchmark is 2^20)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-tte", action="store_true",
                    help="leave out the time-to-eps study (R-MAT 22, learned control variate vs plain) that the "
                         "default run appends to its line")
    ap.add_argument("--workload", choices=["ba", "cv", "grid", "batch", "rb", "group", "roots", "electrical", "solve", "mlp"],
                    default="ba",
                    help="ba: the benchmark line; cv: time to eps = 0.1, learned control variate vs "
                         "plain (R-MAT scale 22); grid: 2048^2 road-like grid, three alphas in one launch; "
                         "batch: 4096 uneven graphs in one launch; rb: Rao-Blackwellised accumulation of "
                         "32 sampled trees of R-MAT (--rmat-scale); group: greedy group forest closeness "
                         "(Algorithm 3) on a weighted BA graph of --group-n vertices, --group-k members; "
                         "roots: forest roots and depths of 152 sampled trees of BA 2^20 plus root counts "
                         "for 64 query vertices (Omega columns); electrical: electrical closeness on G (BA 2^20 "
                         "rooted at its hub, --el-trees trees)")
    ap.add_argument("--el-trees", type=int, default=1024)
    ap.add_argument("--el-estimator", default="visits", choices=["visits", "kirchhoff"],
                    help="electrical workload: r(root, v) from the sampler's visit totals or the Kirchhoff path sums")
    ap.add_argument("--rhs", type=int, default=64, help="right-hand sides of --workload solve")
    ap.add_argument("--grid-side", type=int, default=2048, help="grid workload: side of the grid")
    ap.add_argument("--grid-alphas", default="0.1,1,10", help="grid workload: alphas, comma-separated")
    ap.add_argument("--grid-trees", type=int, default=512, help="grid workload: trees per alpha and step")
    ap.add_argument("--batch-trees", type=int, default=256, help="batch workload: trees per graph and step")
    ap.add_argument("--roots-trees", type=int, default=152, help="roots workload: trees")
    ap.add_argument("--el-order", default="bfs_reverse", choices=["bfs", "bfs_reverse", "id", "id_desc"],
                    help="start order of the rooted sampler (default: the reverse of the root's breadth-first "
                         "order, the library's automatic choice)")
    ap.add_argument("--group-n", type=int, default=16384)
    ap.add_argument("--group-k", type=int, default=64)
    ap.add_argument("--graphs", type=int, default=4096)
    ap.add_argument("--rmat-scale", type=int, default=22)
    ap.add_argument("--seeds", type=int, default=5)
    ap.add_argument("--shape", default="",
                    help="sampler shape 'walkers,regs[,order]' instead of the tuner's choice (profiling runs)")
    return ap.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def profiled_traffic(kname, launched):
    """DRAM bytes per sampler launch from the committed ncu summary, if the
    summary covers the kernel and launch shape that ran and the kernel source
    is unchanged since that capture (else None)."""
    import hashlib
    pop = kname.startswith("k_pop")
    prof = os.path.join(ROOT, "profiles", "k_pop_ba_n2e20_tau1024.md" if pop else "k_wilson_edge_ba_n2e20_tau1024.md")
    src = [os.path.join(ROOT, "paper_2101_06192_gb300", "csrc", f)
           for f in ("fc_pop.cu" if pop else "fc_wilson_edge.cu", "fc_wilson_common.cuh", "fc_internal.cuh")]
    try:
        txt = open(prof).read()
        h = hashlib.sha256(b"".join(open(f, "rb").read() for f in src)).hexdigest()[:16]
        vals = {k.strip(): v.strip() for k, v in (ln.split(":", 1) for ln in txt.splitlines()
                                                   if ln.startswith(("traffic_bytes:", "kernel_src", "launch:")))}
        if vals.get("kernel_src_sha256_16") != h:
            return None
        want = f"{kname} walkers={launched.get('walkers_per_tree')} ctas={launched.get('ctas')}"
        if vals.get("launch") != want:
            return None
        return float(vals["traffic_bytes"])
    except Exception:
        return None


def nvtx_push(name):
    try:
        import torch
        torch.cuda.nvtx.range_push(name)
    except Exception:
        pass


def nvtx_pop():
    try:
        import torch
        torch.cuda.nvtx.range_pop()
    except Exception:
        pass


def load_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


# Algorithmic bytes of the sampler: per walk step (departure) the row info 8 B,
# the selected CSR entry 4 B and the state word read and written 8 B (20 B),
# weighted rows one FP64 slot threshold more (28 B); per vertex and tree one
# retrace read and write of the state word (8 B).
ALG_BYTES_PER_STEP, ALG_BYTES_PER_STEP_WEIGHTED, ALG_BYTES_PER_VERTEX_TREE = 20.0, 28.0, 8.0


def algorithmic_bytes(departures, n, trees, weighted=False):
    per_step = ALG_BYTES_PER_STEP_WEIGHTED if weighted else ALG_BYTES_PER_STEP
    return departures * per_step + ALG_BYTES_PER_VERTEX_TREE * n * trees


def layout_bytes(departures, pops, n, trees, u_edges):
    """Bytes the edge-record kernel's own layout touches: 40 B per departure
    (row info 16, CSR target 4, state read and write 16, next pointer 4), 20 B
    per pop, 20 B per vertex and tree (state clear 16, start order 4), 8 B per
    u*-edge count."""
    return departures * 40 + pops * 20 + trees * n * (16 + 4) + u_edges * 8


class ClockSampler:
    """nvidia-smi clocks/throttle reasons sampled during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                smax = max(smax, float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[3:7]):
                if val.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm)}


def cpu_trees_per_s(g, trees_per_core: int = 4):
    """The oracle's sequential sampler (as it stands), one tree range per host
    core in parallel threads (ctypes releases the GIL)."""
    import concurrent.futures as cf
    from oracle import native
    native.build()
    cores = os.cpu_count() or 1
    total = trees_per_core * cores
    t0 = time.perf_counter()
    with cf.ThreadPoolExecutor(max_workers=cores) as ex:
        futs = [ex.submit(native.wilson, g, ALPHA, 7, trees_per_core, c * trees_per_core, 0, None, False,
                          False, False) for c in range(cores)]
        for f in futs:
            f.result()
    dt = time.perf_counter() - t0
    return total / dt, cores, total, dt


def cpu_single_thread(g, trees: int = 2):
    """The oracle's sequential sampler on one host thread: (trees/s, walk
    steps/s) from its own step counters."""
    from oracle import native
    native.build()
    t0 = time.perf_counter()
    out = native.wilson(g, ALPHA, 7, trees, 10**7, 0, None, False, False, True)
    dt = time.perf_counter() - t0
    return trees / dt, float(out["steps"].sum()) / dt


def bench_config(args, g, world: int) -> dict:
    """The workload description both arms print (identical dicts)."""
    full = args.n_log2 == N_LOG2 and args.tau == TAU
    return {"workload": WORKLOAD if full else
            f"BA n=2^{args.n_log2} m={BA_M} (seed {BA_SEED}) unweighted, alpha={ALPHA:g}, tau={args.tau} "
            "trees/step (profiling case)",
            "n": g.n, "m_edges": g.m, "nnz": g.nnz, "tau": args.tau,
            "l2": "GPU arm: flushed before every timed step (512 MB write)",
            "parallelism": ("one GPU" if world == 1 else
                            f"{world} tree shards: each rank samples its own tau trees, R and C summed by one "
                            "all-reduce")}


def run_reference(args, g):
    """The oracle (sequential Wilson per host thread) on the same workload: each
    step samples a bounded share of the step's trees, 2 per host core, and is
    timed as it stands; value = trees per second over the timed steps."""
    rank, world, _ = dist_env()
    if rank != 0:
        return
    trees_per_core = 2
    times, trees = [], 0
    cores = os.cpu_count() or 1
    total = 0
    for i in range(args.warmup + args.steps):
        rate, cores, total, dt = cpu_trees_per_s(g, trees_per_core)
        if i >= args.warmup:
            times.append(dt)
            trees += total
    value = trees / sum(times)
    st_trees, st_steps = cpu_single_thread(g)
    single = {"trees_per_s": st_trees, "walk_steps_per_s": st_steps, "trees": 2}
    sample = (f"{total} of the step's {args.tau} trees per step ({trees_per_core} per host core, sequential "
              f"Wilson per thread); ms_per_step is the time of that sample")
    line = {
        "metric": "USTs/s", "value": value, "unit": "trees/s", "impl": "reference", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * statistics.mean(times),
        "trees_per_step": total, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "u32/f64", "data": "synthetic", "config": bench_config(args, g, args.gpus),
        "cpu_baseline": {"value": value, "unit": "trees/s", "cores": cores, "kind": "oracle", "sample": sample,
                         "single_thread": single},
        "e2e": {"value": value, "unit": "trees/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def reference_vertices(g, count: int, seed: int):
    """Reference set: stratified by degree decile among non-isolated vertices, plus
    the 256 lowest-degree non-isolated vertices (largest variance)."""
    import numpy as np
    rng = np.random.default_rng(seed)
    d = g.degrees()
    nz = np.nonzero(d > 0)[0]
    order = nz[np.lexsort((nz, d[nz]))]
    low = order[:256]
    rest = np.setdiff1d(nz, low)
    deciles = np.array_split(rest[np.argsort(d[rest], kind="stable")], 10)
    per = max(1, (count - low.size) // 10)
    picks = [low] + [rng.choice(b, size=min(per, b.size), replace=False) for b in deciles if b.size]
    return np.unique(np.concatenate(picks))


def gen_graph(spec):
    """Seeded generator call (runs in a spawned worker process)."""
    import synth
    kind, a = spec
    return {"rmat": synth.rmat, "ba": synth.barabasi_albert}[kind](*a)


def start_generation(specs):
    """Generate graphs in spawned host processes while the GPU works."""
    import concurrent.futures as cf
    import multiprocessing as mp
    ex = cf.ProcessPoolExecutor(max_workers=max(1, min(len(specs), os.cpu_count() or 1)),
                                mp_context=mp.get_context("spawn"))
    return ex, [ex.submit(gen_graph, sp) for sp in specs]


TTE_EPS = 0.1
TRAIN_SCALES = (16, 17, 18)
TRAIN_PER_SCALE = 8


def cv_graph_specs(rmat_scale: int):
    """R-MAT(scale, 16, a = 0.57, b = c = 0.19), seed 4, and the training graphs
    R-MAT 16-18, eight per scale (seeds 100 + i + scale)."""
    return [("rmat", (rmat_scale, 16, 4))] + [("rmat", (sc, 16, 100 + i + sc)) for sc in TRAIN_SCALES
                                             for i in range(TRAIN_PER_SCALE)]


def cv_study(g, train_graphs, seeds: int, rmat_scale: int):
    """Time to max-abs diag(Omega) error <= 0.1 on a 4096-vertex reference set,
    for the plain estimator (Prop. 1), the learned control variate (trained
    network), the same control variate with the untrained network and with the
    feature-free prediction g = p_v (beta = 1), the Rao-Blackwellised estimator
    and the visit estimator (departures / deg*, fc_visit_diag); median GPU time
    over seeds (CUDA events: sampling, features and inference, combination).
    Training time is reported separately."""
    import numpy as np
    import torch
    from paper_2101_06192_gb300 import cvnet, fc, tune
    G = fc.Graph.from_csr(g, [1.0])
    # start order and register variant tuned at the checkpoint scale (tens of
    # trees per launch), untimed; walkers per tree and CTAs per tree stay
    # automatic because the checkpoint launches range from 16 to 1024 trees
    shape = tune.autotune(G, 64)
    G.set_shape(0, 0, 0, shape.get("regs", 0))
    J = reference_vertices(g, 4096, 5)
    Jt = torch.from_numpy(J).cuda()
    TJ = 16384
    ref = G.sample(777_000, TJ, tree_offset=10**6, with_C=False)
    dj, _, _ = G.farness(ref["R"], TJ)
    dj = dj[Jt]
    # spot check of the reference against CG columns (fc_solve) on 4 reference vertices
    sub = J[np.linspace(0, J.size - 1, 4).astype(int)]
    B = torch.zeros((sub.size, g.n), dtype=torch.float64, device="cuda")
    B[torch.arange(sub.size), torch.from_numpy(sub).cuda()] = 1.0
    X, _ = G.solve(B, rel_tol=1e-8)
    om_sub = X[torch.arange(sub.size), torch.from_numpy(sub).cuda()]
    ref_vs_cg = float((dj[torch.from_numpy(np.searchsorted(J, sub)).cuda()] - om_sub).abs().max())
    del B, X
    # training on the smaller R-MAT graphs, targets from the plain estimator
    tt = time.perf_counter()
    train = []
    for i, gs in enumerate(train_graphs):
        Gs = fc.Graph.from_csr(gs, [1.0])
        train.append((Gs, Gs.features(), cvnet.plain_targets(Gs, 4096, seed=100 + i), 0))
    torch.cuda.synchronize()
    targets_s = time.perf_counter() - tt
    tt = time.perf_counter()
    params, hist = cvnet.train(train, steps=500, lr=3e-3, seed=1, log_every=100)
    torch.cuda.synchronize()
    train_s = time.perf_counter() - tt
    for (Gs, _, _, _) in train:
        Gs.close()
    untrained = cvnet.init_params(1)  # the initial parameters of the training run
    checkpoints = [16, 32, 64, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048, 3072, 4096]
    stream = torch.cuda.current_stream()

    def timed(fn):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        r = fn()
        b.record(stream)
        torch.cuda.synchronize()
        return r, a.elapsed_time(b)

    forms = {"plain": None, "cv": params, "cv_untrained": untrained, "cv_p": "p", "rb": None, "visits": None}
    results = {}
    infer_ms = []  # features + MLP forward (fc_vertex_features, fc_mlp_forward)
    for form, prm in forms.items():
        per_seed = []
        for sd in range(seeds):
            R = torch.zeros(g.n, dtype=torch.int32, device="cuda")
            C = torch.zeros(g.n, dtype=torch.int32, device="cuda")
            acc = torch.zeros(g.n, dtype=torch.int64, device="cuda")
            ms = 0.0
            gp = None
            if form.startswith("cv"):
                if prm == "p":
                    # g = 0 clips to p_v: beta = 1, no features, no network
                    gp = torch.zeros(g.n, dtype=torch.float32, device="cuda")
                else:
                    gp, dt = timed(lambda: cvnet.predict(G, prm))
                    if form == "cv":
                        infer_ms.append(dt)
                    ms += dt
            done = 0
            hit = None
            err = None
            vis = torch.zeros(g.n, dtype=torch.int64, device="cuda") if form == "visits" else None
            for cp in checkpoints:
                if form == "visits":
                    # the same trees, departures from each vertex (visit estimate)
                    def vis_step():
                        G.sample(50_000 + 1000 * sd, cp - done, tree_offset=done, R=R, C=C, visits=vis)
                        return G.visit_diag(vis, cp)
                    d, dt = timed(vis_step)
                    ms += dt
                    done = cp
                elif form == "rb":
                    # the same trees, with their parents, summarised by the
                    # Rao-Blackwellised conditional probabilities
                    def rb_step():
                        o = G.sample(50_000 + 1000 * sd, cp - done, tree_offset=done, R=R, C=C, want_parents=True)
                        G.rb_accumulate(o["parents"][0], acc=acc)
                        return G.rb_diag(acc, cp)
                    d, dt = timed(rb_step)
                    ms += dt
                    done = cp
                else:
                    _, dt = timed(lambda: G.sample(50_000 + 1000 * sd, cp - done, tree_offset=done, R=R, C=C))
                    ms += dt
                    done = cp
                    if gp is not None:
                        (d, _, _), dt = timed(lambda: G.farness(R, cp, C=C, g_pred=gp))
                    else:
                        (d, _, _), dt = timed(lambda: G.farness(R, cp))
                    ms += dt
                err = float((d[Jt] - dj).abs().max())
                if err <= TTE_EPS:
                    hit = {"trees": cp, "ms": ms, "max_err": err}
                    break
            per_seed.append(hit or {"trees": None, "ms": ms, "max_err": err})
        ok = [r for r in per_seed if r["trees"] is not None]
        results[form] = {
            "median_ms": statistics.median(r["ms"] for r in ok) if len(ok) == len(per_seed) else None,
            "median_trees": statistics.median(r["trees"] for r in ok) if len(ok) == len(per_seed) else None,
            "runs": per_seed,
        }
    G.close()
    med = {f: results[f]["median_ms"] for f in forms}
    summary = {
        "eps": TTE_EPS, "unit": "ms", "seeds": seeds,
        "workload": f"R-MAT scale {rmat_scale} ef 16 (0.57,0.19,0.19) seed 4, alpha=1",
        "plain_ms": med["plain"], "cv_ms": med["cv"], "cv_untrained_ms": med["cv_untrained"],
        "cv_p_ms": med["cv_p"], "rb_ms": med["rb"], "visits_ms": med["visits"],
        "trees": {f: results[f]["median_trees"] for f in forms},
        "speedup_cv_over_plain": (med["plain"] / med["cv"]) if med["cv"] and med["plain"] else None,
        "speedup_cv_over_untrained": (med["cv_untrained"] / med["cv"]) if med["cv"] and med["cv_untrained"] else None,
        "speedup_cv_over_p": (med["cv_p"] / med["cv"]) if med["cv"] and med["cv_p"] else None,
        "reference_set": {"vertices": int(J.size), "plain_trees": TJ, "reference_vs_cg_max_abs": ref_vs_cg},
        "train": {"graphs": f"R-MAT scale {TRAIN_SCALES[0]}-{TRAIN_SCALES[-1]} x{TRAIN_PER_SCALE}, plain targets "
                            "tau=4096", "steps": 500, "loss_first_last": [hist[0][1], hist[-1][1]],
                  "seconds": train_s, "target_seconds": targets_s},
        # features + forward pass per vertex: about 1.55 kFLOP FP32 (128 hidden
        # units x (4 FMAs + bias + relu) + 128 FMAs + the sigmoid); CUDA-core
        # FP32 peak 152 SMs x 128 lanes x 2 x 2.07 GHz = 80.5 TFLOP/s
        "cv_inference": {"ms": statistics.median(infer_ms) if infer_ms else None,
                         "tflops": (1.55e3 * g.n / (statistics.median(infer_ms) / 1000.0) / 1e12) if infer_ms else None,
                         "fp32_peak_tflops": 80.5, "bytes_per_vertex": 16 + 4},
        "sampler_shape": shape,
    }
    return summary, results


def run_cv(args):
    """Time to max-abs diag(Omega) error <= 0.1, learned control variate vs plain
    estimator and the ablations, R-MAT(scale, 16, a=0.57, b=c=0.19), alpha = 1."""
    import torch
    torch.cuda.set_device(0)
    t0 = time.perf_counter()
    ex, futs = start_generation(cv_graph_specs(args.rmat_scale))
    graphs = [f.result() for f in futs]
    ex.shutdown()
    gen_s = time.perf_counter() - t0
    g = graphs[0]
    summary, results = cv_study(g, graphs[1:], args.seeds, args.rmat_scale)
    line = {
        "metric": "time to eps=0.1 max-abs diag(Omega) error", "unit": "ms", "higher_is_better": False,
        "value": summary["cv_ms"], "time_to_eps": summary,
        "config": {"workload": summary["workload"], "n": g.n, "m_edges": g.m, "gen_seconds": gen_s},
        "dtype": "u32/f64 (MLP bf16/fp32)", "data": "synthetic", "runs": results,
    }
    print(json.dumps(line), flush=True)


def run_grid(args):
    """Road-like graph, three alphas in one persistent launch: 2048 x 2048
    4-neighbour grid, 10% of edges deleted, 1% diagonal shortcuts, weights
    U[1, 10] FP32; alpha in {0.1, 1, 10}, 512 trees each per step."""
    import torch
    import synth
    from paper_2101_06192_gb300 import fc, tune
    torch.cuda.set_device(0)
    side = args.grid_side
    g = synth.perturbed_grid(side, side, 3)
    alphas = [float(a) for a in args.grid_alphas.split(",")]
    tau = args.grid_trees
    G = fc.Graph.from_csr(g, alphas)
    if args.shape:  # fixed shape 'walkers,regs[,order]' (profiling cases)
        parts = args.shape.split(",")
        shape = {"walkers": int(parts[0]), "regs": int(parts[1]), "order": parts[2] if len(parts) > 2 else "auto"}
        tune.apply(G, shape)
    else:
        shape = tune.autotune(G, tau)
    stream = torch.cuda.current_stream()
    R = torch.zeros(len(alphas) * g.n, dtype=torch.int32, device="cuda")
    for i in range(max(1, args.warmup)):
        G.sample(100 + i, 32, R=R.zero_(), with_C=False)
    times, stats = [], []
    clocks = ClockSampler(0)
    clocks.start()
    nvtx_push("timed")
    for i in range(args.steps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        R.zero_()
        a.record(stream)
        G.sample(200 + i, tau, R=R, with_C=False)
        for ai in range(len(alphas)):
            G.farness(R, tau, alpha_idx=ai)
        b.record(stream)
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
        stats.append(G.sampler_stats())
    nvtx_pop()
    clk = clocks.stop()
    ms = statistics.mean(times)
    pops = statistics.mean(s[0] for s in stats)
    deps = statistics.mean(s[1] for s in stats)
    n_trees = len(alphas) * tau
    alg_bytes = algorithmic_bytes(deps, g.n, n_trees, weighted=True)
    layout = layout_bytes(deps, pops, g.n, n_trees, 0)
    peaks, peak_kind = load_peaks()
    achieved = alg_bytes / (ms / 1000.0) / 1e9
    line = {
        "metric": "USTs/s", "value": n_trees / (ms / 1000.0), "unit": "trees/s", "ms_per_step": ms,
        "higher_is_better": True, "steps": args.steps, "dtype": "u32/f64", "data": "synthetic",
        "config": {"workload": f"grid {side}^2, 10% deleted, 1% diagonals, w~U[1,10] fp32, alpha "
                               f"{{{args.grid_alphas}}} x {tau} trees",
                   "n": g.n, "m_edges": g.m, "shape": shape},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": float(peaks.get("hbm_gbs", 6800.0)),
                     "unit": "GB/s", "frac": achieved / float(peaks.get("hbm_gbs", 6800.0)),
                     "peak_source": peak_kind, "departures_per_step": deps, "pops_per_step": pops,
                     "algorithmic_bytes": alg_bytes, "layout_bytes": layout,
                     "layout_frac": layout / (ms / 1000.0) / 1e9 / float(peaks.get("hbm_gbs", 6800.0))},
        "clocks": clk,
    }
    G.close()
    print(json.dumps(line), flush=True)


def run_batch(args):
    """Uneven batch: graphs with n log-uniform in [100, 50000] (half BA m in
    2..8, half perturbed grids), alpha log-uniform in [0.1, 10], 256 trees of
    every graph in one persistent launch, plain and learned-CV combination."""
    import numpy as np
    import torch
    import synth
    from paper_2101_06192_gb300 import cvnet, fc, tune
    torch.cuda.set_device(0)
    t0 = time.perf_counter()
    graphs, alphas = synth.uneven_batch(args.graphs, 5)
    u, offs = synth.union(graphs)
    gen_s = time.perf_counter() - t0
    G = fc.Graph.batch(u, offs, alphas)
    tau = args.batch_trees
    shape = tune.autotune(G, tau, probe_trees=32)  # start order and shape, untimed
    # control-variate network: trained on small R-MAT graphs (untimed)
    train = []
    for sc, sd in ((12, 100), (13, 101), (14, 102)):
        gs = synth.rmat(sc, 16, sd)
        Gs = fc.Graph.from_csr(gs, [1.0])
        train.append((Gs, Gs.features(), cvnet.plain_targets(Gs, 2048, seed=sd), 0))
    params, _ = cvnet.train(train, steps=300, lr=3e-3, seed=1)
    for (Gs, _, _, _) in train:
        Gs.close()
    stream = torch.cuda.current_stream()
    R = torch.zeros(u.n, dtype=torch.int32, device="cuda")
    C = torch.zeros(u.n, dtype=torch.int32, device="cuda")
    G.sample(1, 4, R=R, C=C)  # warm-up
    times = []
    nvtx_push("timed")
    for i in range(args.steps):
        R.zero_()
        C.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        G.sample(300 + i, tau, R=R, C=C)
        gp = cvnet.predict(G, params)
        d_cv, far, clo = G.farness(R, tau, C=C, g_pred=gp)
        b.record(stream)
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    nvtx_pop()
    lat = G.batch_latency_ms()
    d_plain, _, _ = G.farness(R, tau)
    # accuracy on the small graphs; reference: diag(Omega) from the library's CG
    # solve of (I + alpha L) X = I on each graph (independent of the sampler)
    dp, dc = d_plain.cpu().numpy(), d_cv.cpu().numpy()
    small = [i for i, g in enumerate(graphs) if g.n <= 1500][:40]
    ep, ec = [], []
    for i in small:
        Gi = fc.Graph.from_csr(graphs[i], [float(alphas[i])])
        X, _ = Gi.solve(torch.eye(graphs[i].n, dtype=torch.float64, device="cuda"), rel_tol=1e-10)
        om = torch.diagonal(X).cpu().numpy()
        Gi.close()
        a_, b_ = offs[i], offs[i + 1]
        ep.append(float(np.max(np.abs(dp[a_:b_] - om))))
        ec.append(float(np.max(np.abs(dc[a_:b_] - om))))
    ms = statistics.mean(times)
    line = {
        "metric": "USTs/s", "value": args.graphs * tau / (ms / 1000.0), "unit": "graph-trees/s",
        "ms_per_step": ms, "higher_is_better": True, "steps": args.steps, "dtype": "u32/f64", "data": "synthetic",
        "config": {"workload": f"{args.graphs} graphs, n log-uniform [100, 50000], half BA half grid, "
                               f"alpha log-uniform [0.1, 10], {tau} trees each + learned CV",
                   "total_vertices": int(u.n), "total_edges": int(u.m), "gen_seconds": gen_s,
                   "sampler_shape": shape},
        "latency_ms": {"p50": float(np.percentile(lat, 50)), "p99": float(np.percentile(lat, 99)),
                       "max": float(lat.max())},
        "max_abs_diag_err_small_graphs": {"graphs": len(small), "plain_median": float(np.median(ep)),
                                          "cv_median": float(np.median(ec))},
    }
    G.close()
    print(json.dumps(line), flush=True)


def run_rb(args):
    """Rao-Blackwellised accumulation (fc_rb_accumulate) of 32 trees sampled
    with their parents on R-MAT(scale, 16), alpha = 1: (tree, vertex) pairs per
    second of the accumulation alone, inputs resident, L2 flushed before each
    timed call."""
    import torch
    import synth
    from paper_2101_06192_gb300 import fc
    torch.cuda.set_device(0)
    g = synth.rmat(args.rmat_scale, 16, 4)
    G = fc.Graph.from_csr(g, [1.0])
    T = 32
    par = G.sample(6, T, want_parents=True)["parents"][0]
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        G.rb_accumulate(par)
    torch.cuda.synchronize()
    clocks = ClockSampler(0)
    clocks.start()
    ms = []
    nvtx_push("timed")
    for _ in range(args.steps):
        flush.zero_()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        G.rb_accumulate(par)
        b.record(stream)
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    nvtx_pop()
    clk = clocks.stop()
    t = statistics.mean(ms) / 1000.0
    n, nnz = g.n, int(g.rowptr[-1])
    # algorithmic bytes per call: parents read, CSR rows read once, one
    # neighbour test per (tree, CSR entry) reading a 4-byte preorder number,
    # one u64 total per vertex
    alg = 4 * T * n + (4 * nnz + 8 * (n + 1)) + 4 * T * nnz + 8 * n
    peaks, peak_kind = load_peaks()
    peak = float(peaks.get("hbm_gbs", 6800.0))
    line = {"metric": "tree-vertices/s (Rao-Blackwellised accumulation)", "value": T * n / t,
            "unit": "tree-vertices/s", "ms_per_call": statistics.mean(ms), "steps": args.steps,
            "warmup": args.warmup, "higher_is_better": True, "dtype": "u64 fixed point / f64",
            "data": "synthetic", "config": {"workload": f"R-MAT scale {args.rmat_scale} ef 16, alpha=1, 32 trees "
                                                        "with parents, one chunk", "n": n, "nnz": nnz,
                                            "l2": "flushed before every timed call (512 MB write)"},
            "roofline": {"bound": "hbm", "achieved": alg / t / 1e9, "peak": peak, "unit": "GB/s",
                         "frac": alg / t / 1e9 / peak, "traffic": None, "kernel": "k_rb",
                         "algorithmic_bytes": alg, "peak_source": peak_kind},
            "clocks": clk}
    G.close()
    print(json.dumps(line), flush=True)


def run_group(args):
    """Greedy group forest closeness (fc_group_closeness, Algorithm 3) on a
    weighted BA graph (m = 4, weights U[0.5, 3]), alpha = 1: the whole call
    (forest matrix by CG, the grounded inverse, k - 1 greedy passes) and the
    greedy part alone (a k = 1 call subtracted)."""
    import numpy as np
    import torch
    import synth
    from paper_2101_06192_gb300 import fc
    torch.cuda.set_device(0)
    n, k = args.group_n, args.group_k
    base = synth.barabasi_albert(n, 4, 7)
    u, v, _ = base.edges()
    rng = np.random.default_rng(8)
    g = synth.from_edges(n, u, v, rng.uniform(0.5, 3.0, u.size).astype(np.float32))
    G = fc.Graph.from_csr(g, [1.0])
    stream = torch.cuda.current_stream()

    def timed(kk):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        S, far = G.group_closeness(kk)
        b.record(stream)
        torch.cuda.synchronize()
        return a.elapsed_time(b), S, far

    for _ in range(max(1, args.warmup)):
        timed(k)
    clocks = ClockSampler(0)
    clocks.start()
    nvtx_push("timed")
    full = [timed(k) for _ in range(args.steps)]
    one = [timed(1)[0] for _ in range(args.steps)]
    nvtx_pop()
    clk = clocks.stop()
    t_full = statistics.median(x[0] for x in full)
    t_one = statistics.median(one)
    per_step = (t_full - t_one) / max(1, k - 1)
    S, far = full[-1][1].cpu().numpy(), full[-1][2].cpu().numpy()
    n1 = n + 1
    pass_bytes = 16.0 * n1 * n1  # M read and written once per greedy step
    peaks, peak_kind = load_peaks()
    peak = float(peaks.get("hbm_gbs", 6800.0))
    # the pass does two FP64 FMAs per entry (downdate, squared norm) and is
    # bound by the FP64 pipe: 152 SMs x 2 FP64 FMA per SM-clock x 2.07 GHz
    # = 1.26 TFLOP/s (4 flops per entry)
    fp64_peak = 152 * 2 * 2 * 2.07e9 / 1e12
    flops = 4.0 * n1 * n1
    achieved = flops / (per_step / 1000.0) / 1e12
    line = {"metric": "group forest closeness, greedy steps/s (Algorithm 3)", "value": 1000.0 / per_step,
            "unit": "steps/s", "ms_total": t_full, "ms_setup_k1": t_one, "ms_per_greedy_step": per_step,
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": f"weighted BA n={n} m=4 w~U[0.5,3], alpha=1, k={k}", "n": n, "k": k,
                       "nnz": int(g.rowptr[-1])},
            "roofline": {"bound": "alu", "achieved": achieved, "peak": fp64_peak, "unit": "TFLOP/s (FP64)",
                         "frac": achieved / fp64_peak, "traffic": None, "kernel": "k_grp_pass",
                         "peak_source": "derived: 152 SMs x 2 FP64 FMA/clk x 2.07 GHz",
                         "hbm": {"bytes_per_step": pass_bytes, "achieved_gbs": pass_bytes / (per_step / 1000.0) / 1e9,
                                 "peak_gbs": peak, "frac": pass_bytes / (per_step / 1000.0) / 1e9 / peak,
                                 "peak_source": peak_kind}},
            "group_head": S[:8].tolist(), "farness_first_last": [float(far[0]), float(far[-1])],
            "clocks": clk}
    if not args.no_cpu_baseline:
        from oracle import group as ogroup
        ns = 2048
        us, vs, _ = synth.barabasi_albert(ns, 4, 7).edges()
        gs = synth.from_edges(ns, us, vs, np.random.default_rng(9).uniform(0.5, 3.0, us.size).astype(np.float32))
        t0 = time.perf_counter()
        ogroup.greedy(gs, 1.0, 32)
        dt = time.perf_counter() - t0
        line["cpu_baseline"] = {"value": 31.0 / dt, "unit": "steps/s", "cores": os.cpu_count(), "kind": "oracle",
                                "sample": f"Algorithm 3 on weighted BA n={ns}, k=32 (numpy FP64, {dt:.2f} s "
                                          "including the dense pseudo-inverse and inverse)"}
    G.close()
    print(json.dumps(line), flush=True)


def run_roots(args):
    """Forest roots and depths of sampled trees on the benchmark graph (BA
    n = 2^20, m = 8), 152 trees: one call of the sampler
    (fc_sample_usts_forest), against sampling with parents followed by
    pointer jumping (fc_tree_roots); and root counts of 64 query vertices
    (fc_root_counts: columns of Omega from the same trees).  L2 flushed before
    each timed call."""
    import numpy as np
    import torch
    import synth
    from paper_2101_06192_gb300 import fc
    torch.cuda.set_device(0)
    g = synth.barabasi_albert(1 << args.n_log2, BA_M, BA_SEED)
    G = fc.Graph.from_csr(g, [ALPHA])
    T = args.roots_trees
    queries = torch.from_numpy(np.linspace(0, g.n - 1, 64).astype(np.int64)).cuda()
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream()

    def timed(fn):
        flush.zero_()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        r = fn()
        b.record(stream)
        torch.cuda.synchronize()
        return a.elapsed_time(b), r

    for _ in range(args.warmup):
        par = G.sample(11, T, want_parents=True, with_C=False)["parents"][0].contiguous()
        roots, depth = fc.tree_roots(par)
        fc.root_counts(roots, queries)
        G.sample(11, T, want_roots=True, with_C=False)
    ms_sp, ms_roots, ms_counts, ms_fused = [], [], [], []
    nvtx_push("timed")
    for _ in range(args.steps):
        t, out = timed(lambda: G.sample(11, T, want_parents=True, with_C=False))
        ms_sp.append(t)
        par = out["parents"][0].contiguous()
        t, (roots, depth) = timed(lambda: fc.tree_roots(par))
        ms_roots.append(t)
        t, _ = timed(lambda: fc.root_counts(roots, queries))
        ms_counts.append(t)
        t, fused = timed(lambda: G.sample(11, T, want_roots=True, with_C=False))
        ms_fused.append(t)
    nvtx_pop()
    same = bool(torch.equal(fused["roots"][0], roots) and torch.equal(fused["depths"][0], depth))
    n = g.n
    t_r = statistics.median(ms_roots) / 1000.0
    t_f = statistics.median(ms_fused) / 1000.0
    # algorithmic bytes of fc_tree_roots: parents read, roots and depths
    # written (4 B each per tree and vertex)
    alg = 12.0 * T * n
    peaks, peak_kind = load_peaks()
    peak = float(peaks.get("hbm_gbs", 6800.0))
    line = {"metric": "tree-vertices/s (trees sampled with forest roots and depths)", "value": T * n / t_f,
            "unit": "tree-vertices/s", "ms_sample_with_forest": 1000.0 * t_f,
            "ms_sample_with_parents": statistics.median(ms_sp), "ms_tree_roots": 1000.0 * t_r,
            "ms_root_counts_64": statistics.median(ms_counts), "fused_equals_pointer_jumping": same,
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "dtype": "i32",
            "data": "synthetic",
            "config": {"workload": f"BA n=2^{args.n_log2} m={BA_M}, alpha={ALPHA:g}, {T} trees, 64 queries",
                       "l2": "flushed before every timed call (512 MB write)"},
            "roofline": {"bound": "hbm", "achieved": alg / t_r / 1e9, "peak": peak, "unit": "GB/s",
                         "frac": alg / t_r / 1e9 / peak, "traffic": None, "kernel": "k_roots",
                         "algorithmic_bytes": alg, "peak_source": peak_kind},
            "max_depth": int(depth.max().item())}
    G.close()
    print(json.dumps(line), flush=True)


def run_electrical(args):
    """Electrical closeness on G (Sec. 3 insights (i)-(iii), Eq. 2): BA n = 2^20,
    m = 8 rooted at its largest hub; one step = build G rooted at the pivot
    (with its BFS tree), sample tau spanning trees, estimate r(root, v) -- by
    default from the sampler's visit totals (Green's function), with
    --el-estimator kirchhoff from the parents by the Kirchhoff path sums
    (fc_resistance_accumulate) -- the pivot column of L^+ (fc_laplacian_solve)
    and the combination (fc_electrical_closeness).  Untimed: both estimates
    from the same 256 trees against L^+[v, v] of reference vertices."""
    import numpy as np
    import torch
    import synth
    from paper_2101_06192_gb300 import fc
    torch.cuda.set_device(0)
    g = synth.barabasi_albert(1 << args.n_log2, BA_M, BA_SEED)
    root = int(np.argmax(g.degrees()))
    tau = args.el_trees
    n = g.n
    stream = torch.cuda.current_stream()
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    e = torch.zeros(n, dtype=torch.float64, device="cuda")
    e[root] = 1.0
    out = {}

    def step(seed, ev=None):
        G = fc.Graph.rooted(g, root)
        if args.el_order != "bfs_reverse":
            # on a rooted graph the order array holds the breadth-first order
            G.set_start_order({"bfs": 0, "id": 2, "id_desc": 3}[args.el_order])
        if ev:
            ev[0].record(stream)
        kir = args.el_estimator == "kirchhoff"
        o = G.sample(seed, tau, want_parents=kir, want_visits=not kir, with_C=False)
        if ev:
            ev[1].record(stream)
        acc = G.resistance_accumulate(o["parents"][0]) if kir else None
        if ev:
            ev[2].record(stream)
        x, it = G.laplacian_solve(e, rel_tol=1e-9)
        if ev:
            ev[3].record(stream)
        r, d, far, clo = G.electrical_closeness(acc, tau, x, visits=o["visits"])
        out.update(diag=d, iters=it, depth=int(G.bfs_tree()[1].max().item()), stats=G.sampler_stats())
        G.close()
        return clo

    for i in range(args.warmup):
        step(100 + i)
    torch.cuda.synchronize()
    clocks = ClockSampler(0)
    clocks.start()
    tot, parts = [], []
    nvtx_push("timed")
    for i in range(args.steps):
        flush.zero_()
        torch.cuda.synchronize()
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(6)]
        evs[0].record(stream)
        step(200 + i, ev=evs[1:5])
        evs[5].record(stream)
        torch.cuda.synchronize()
        tot.append(evs[0].elapsed_time(evs[5]))
        parts.append([evs[k].elapsed_time(evs[k + 1]) for k in range(5)])
    nvtx_pop()
    clk = clocks.stop()
    ms = statistics.mean(tot)
    pm = [statistics.mean(p[k] for p in parts) for k in range(5)]
    # accuracy: L^+[v, v] of reference vertices by Laplacian solves (exact to 1e-10)
    J = reference_vertices(g, 64, 7)
    Gj = fc.Graph.rooted(g, root)
    B = torch.zeros(J.size, n, dtype=torch.float64, device="cuda")
    Jt = torch.from_numpy(J).cuda()
    B[torch.arange(J.size, device="cuda"), Jt] = 1.0
    X, _ = Gj.laplacian_solve(B, rel_tol=1e-10)
    exact = X[torch.arange(J.size, device="cuda"), Jt]
    depth_sum = float(Gj.bfs_tree()[1].to(torch.float64).sum().item())
    # both estimators on the same 256 trees (untimed)
    tc = 256
    o = Gj.sample(99, tc, want_parents=True, want_visits=True, with_C=False)
    xj, _ = Gj.laplacian_solve(e, rel_tol=1e-10)
    cmp = {}
    for name, acc_, vis_ in (("kirchhoff", Gj.resistance_accumulate(o["parents"][0]), None),
                             ("visits", None, o["visits"])):
        _, dd, _, _ = Gj.electrical_closeness(acc_, tc, xj, visits=vis_)
        ee = (dd[Jt] - exact).abs()
        cmp[name] = {"max_abs_err": float(ee.max()), "mean_abs_err": float(ee.mean())}
    del o
    Gj.close()
    err = (out["diag"][Jt] - exact).abs()
    peaks, peak_kind = load_peaks()
    peak = float(peaks.get("hbm_gbs", 6800.0))
    # algorithmic bytes of the path sums: parents read once (4 B per tree and
    # vertex) and, per tree and breadth-first step, the parent of the edge's
    # upper end (4 B); totals 8 B per vertex per chunk of 32 trees
    acc_bytes = 4.0 * tau * n + 4.0 * tau * depth_sum + 8.0 * n * math.ceil(tau / 32)
    acc_s = max(pm[2], 1e-6) / 1000.0
    if args.el_estimator == "kirchhoff":
        roofline = {"bound": "hbm", "kernel": "k_rb<1> (resistance path sums)",
                    "achieved": acc_bytes / acc_s / 1e9, "peak": peak, "unit": "GB/s",
                    "frac": acc_bytes / acc_s / 1e9 / peak, "algorithmic_bytes": acc_bytes,
                    "peak_source": peak_kind, "traffic": None}
    else:  # the sampler dominates: 20 B per walk step + 8 B per vertex and tree
        smp_bytes = algorithmic_bytes(out["stats"][1], n, tau)
        smp_s = pm[1] / 1000.0
        roofline = {"bound": "hbm", "kernel": "k_pop on G rooted at the hub (+ visit totals)",
                    "achieved": smp_bytes / smp_s / 1e9, "peak": peak, "unit": "GB/s",
                    "frac": smp_bytes / smp_s / 1e9 / peak, "algorithmic_bytes": smp_bytes,
                    "peak_source": peak_kind, "traffic": None}
    line = {
        "metric": "USTs/s (electrical closeness on G)", "value": tau / (ms / 1000.0), "unit": "trees/s",
        "ms_per_step": ms, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True,
        "dtype": "u32/i64 fixed point/f64", "data": "synthetic",
        "config": {"workload": f"BA n=2^{args.n_log2} m={BA_M} (seed {BA_SEED}) rooted at its largest hub "
                               f"(degree {int(g.degrees()[root])}), {tau} trees/step",
                   "start_order": args.el_order,
                   "n": n, "m_edges": g.m, "root": root, "bfs_depth_max": out["depth"],
                   "bfs_depth_mean": depth_sum / n,
                   "l2": "flushed before every timed step (512 MB write)"},
        "ms_build": pm[0], "ms_sample": pm[1], "ms_accumulate": pm[2], "ms_solve": pm[3], "ms_combine": pm[4],
        "cg_iterations": out["iters"],
        "departures_per_step": out["stats"][1],
        "accuracy": {"reference_vertices": int(J.size), "max_abs_err_diag_Lplus": float(err.max()),
                     "mean_abs_err": float(err.mean()), "estimators_256_trees": cmp},
        "estimator": args.el_estimator,
        "roofline": roofline,
        "clocks": clk,
    }
    print(json.dumps(line), flush=True)


def run_solve(args):
    """CG on I + alpha L (fc_solve: Jacobi-preconditioned FP32 inner CG, FP64
    residual and refinement to 1e-9) with --rhs right-hand sides e_v of
    degree-stratified reference vertices: on BA n = 2^20, m = 8 (alpha = 1) and
    on the 2048^2 road-like grid (weights U[1, 10], alpha = 1).  Roofline:
    algorithmic bytes of one inner iteration (SpMV: row pointers 8 B per row,
    column index 4 B and weight 4 B per entry, 4 B per entry and right-hand
    side for the gathered vector; the vector updates: 48 B per vertex and
    right-hand side) times the inner iterations, over the solve's time."""
    import numpy as np
    import torch
    import synth
    from paper_2101_06192_gb300 import fc
    torch.cuda.set_device(0)
    stream = torch.cuda.current_stream()
    peaks, peak_kind = load_peaks()
    peak = float(peaks.get("hbm_gbs", 6800.0))
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    results = []
    for name, g in (("BA n=2^20 m=8 (seed 2)", synth.barabasi_albert(1 << N_LOG2, BA_M, BA_SEED)),
                    ("grid 2048^2 (seed 3), w~U[1,10]", synth.perturbed_grid(2048, 2048, 3))):
        G = fc.Graph.from_csr(g, [1.0])
        m = args.rhs
        J = reference_vertices(g, m, 5)[:m]
        m = int(J.size)
        B = torch.zeros((m, g.n), dtype=torch.float64, device="cuda")
        B[torch.arange(m, device="cuda"), torch.from_numpy(J).cuda()] = 1.0
        for _ in range(max(1, args.warmup)):
            G.solve(B, rel_tol=1e-9)
        ms, its = [], []
        nvtx_push("timed")
        for _ in range(args.steps):
            flush.zero_()
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            X, it = G.solve(B, rel_tol=1e-9)
            b.record(stream)
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
            its.append(it)
        nvtx_pop()
        n, nnz = g.n, g.nnz
        wbytes = 4 if g.w is not None else 0
        spmv = 8.0 * (n + 1) + (4.0 + wbytes) * nnz + 4.0 * m * nnz
        it_bytes = spmv + 48.0 * m * n
        t = statistics.median(ms) / 1000.0
        it = statistics.median(its)
        results.append({"graph": name, "n": n, "nnz": nnz, "rhs": m, "ms": statistics.median(ms),
                        "inner_iterations": it, "ms_per_iteration": 1000.0 * t / max(1, it),
                        "spmv_bytes_per_iteration": spmv, "bytes_per_iteration": it_bytes,
                        "achieved_gbs": it_bytes * it / t / 1e9, "frac": it_bytes * it / t / 1e9 / peak})
        G.close()
        del B, X
    line = {"metric": "CG on I + alpha L, achieved algorithmic GB/s", "value": results[0]["achieved_gbs"],
            "unit": "GB/s", "higher_is_better": True, "steps": args.steps, "warmup": args.warmup,
            "dtype": "f32 inner / f64 residual", "data": "synthetic", "results": results,
            "roofline": {"bound": "hbm",
                         "kernel": ("CG inner iteration (k_cg1: edge-tile SpMV + vector phases, one cooperative "
                                    "launch per refinement step)" if args.rhs == 1 else
                                    "CG inner iteration (k_il_spmv + vector kernels)"),
                         "achieved": results[0]["achieved_gbs"], "peak": peak, "unit": "GB/s",
                         "frac": results[0]["frac"], "traffic": None, "peak_source": peak_kind},
            "config": {"workload": f"fc_solve, {args.rhs} right-hand sides e_v, rel_tol 1e-9, alpha=1",
                       "l2": "flushed before every timed solve (512 MB write)"}}
    print(json.dumps(line), flush=True)


def run_mlp(args):
    """Training step of the control-variate network (fc_mlp_loss_grad_acc per
    graph, then fc_mlp_adam) on R-MAT scale 16, 17 and 18 (one graph each,
    plain-estimator targets from 512 trees): graph-steps per second; about
    3 kFLOP FP32 per vertex (forward 1.55 k, backward 1.5 k)."""
    import torch
    import synth
    from paper_2101_06192_gb300 import cvnet, fc
    torch.cuda.set_device(0)
    data = []
    nv = 0
    for i, sc in enumerate((16, 17, 18)):
        g = synth.rmat(sc, 16, 100 + sc)
        G = fc.Graph.from_csr(g, [1.0])
        data.append((G, G.features(), cvnet.plain_targets(G, 512, seed=i), 0))
        nv += g.n
    params = cvnet.init_params(1)
    cvnet.train(data, steps=max(1, args.warmup), lr=1e-3, params=params)
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    nvtx_push("timed")
    a.record(stream)
    cvnet.train(data, steps=args.steps, lr=1e-3, params=params)
    b.record(stream)
    torch.cuda.synchronize()
    nvtx_pop()
    ms = a.elapsed_time(b) / args.steps
    tflops = 3.05e3 * nv / (ms / 1000.0) / 1e12
    line = {"metric": "control-variate training steps/s (3 graphs per step)", "value": 1000.0 / ms,
            "unit": "steps/s", "ms_per_step": ms, "steps": args.steps, "warmup": args.warmup,
            "higher_is_better": True, "dtype": "bf16 weights / fp32", "data": "synthetic",
            "config": {"workload": "R-MAT scale 16, 17, 18 (ef 16), 4->128->1 MLP", "vertices": nv},
            "roofline": {"bound": "alu", "achieved": tflops, "peak": 80.5, "unit": "TFLOP/s (FP32)",
                         "frac": tflops / 80.5, "kernel": "k_mlp_grad",
                         "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 x 2.07 GHz", "traffic": None}}
    for (G, _, _, _) in data:
        G.close()
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.workload == "mlp":
        if rank == 0:
            run_mlp(args)
        return
    if args.workload == "solve":
        if rank == 0:
            run_solve(args)
        return
    if args.workload == "electrical":
        if rank == 0:
            run_electrical(args)
        return
    if args.workload == "roots":
        if rank == 0:
            run_roots(args)
        return
    if args.workload == "group":
        if rank == 0:
            run_group(args)
        return
    if args.workload == "rb":
        if rank == 0:
            run_rb(args)
        return
    if args.workload == "batch":
        if rank == 0:
            run_batch(args)
        return
    if args.workload == "grid":
        if rank == 0:
            run_grid(args)
        return
    if args.workload == "cv":
        if rank == 0:
            run_cv(args)
        return
    import synth
    full = args.n_log2 == N_LOG2 and args.tau == TAU
    # time to eps (R-MAT 22, learned control variate vs plain): its graphs are
    # generated by host processes while the GPU runs the timed steps
    tte_gen = None
    if args.impl == "ours" and rank == 0 and world == 1 and full and not args.no_tte:
        tte_gen = start_generation(cv_graph_specs(args.rmat_scale))
    g = synth.barabasi_albert(1 << args.n_log2, BA_M, BA_SEED)
    if args.impl == "reference":
        run_reference(args, g)
        return

    import torch
    from paper_2101_06192_gb300 import fc, shard
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    tau = args.tau
    n, nnz = g.n, g.nnz
    rowptr_d = torch.from_numpy(g.rowptr).to(dev)
    colidx_d = torch.from_numpy(g.colidx).to(dev)
    rowptr_h = torch.from_numpy(g.rowptr).pin_memory()
    colidx_h = torch.from_numpy(g.colidx).pin_memory()
    # the results read back in the end-to-end steps land in pinned host buffers
    clo_h = torch.empty(n, dtype=torch.float64).pin_memory()
    top_h = torch.empty(TOPK, dtype=torch.int32).pin_memory()
    R = torch.zeros(n, dtype=torch.int32, device=dev)
    C = torch.zeros(n, dtype=torch.int32, device=dev)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream()
    # weak scaling: every rank samples its own tau trees of a world * tau run
    tree_offset, _ = shard.tree_range(rank, world, world * tau)
    shape = {}
    launched = {}
    last_diag = [None]
    from paper_2101_06192_gb300 import tune

    def step(seed, host_inputs=False, samp_ev=None, stats=None):
        if host_inputs:
            G = fc.Graph(rowptr_h.numpy(), colidx_h.numpy(), None, [ALPHA])
        else:
            G = fc.Graph(rowptr_d, colidx_d, None, [ALPHA])
        tune.apply(G, shape)
        R.zero_()
        C.zero_()
        if samp_ev is not None:
            samp_ev[0].record(stream)
        G.sample(seed, tau, tree_offset=tree_offset, R=R, C=C)
        if samp_ev is not None:
            samp_ev[1].record(stream)
        if stats is not None:
            stats.append(G.sampler_stats())
            launched.update(kernel=G.last_kernel(), cluster=G.last_cluster(), **G.last_shape())
        if world > 1:
            shard.allreduce_counts(R, C)  # the one exchange of the sharded estimator
        x, _ = G.pivot_solve(rel_tol=1e-9)
        diag, far, clo = G.farness(R, world * tau, x_pivot=x)
        top = fc.top_k(diag, TOPK)
        G.close()
        last_diag[0] = diag
        if host_inputs:
            clo_h.copy_(clo, non_blocking=True)
            top_h.copy_(top, non_blocking=True)
            torch.cuda.current_stream().synchronize()
            return clo_h, top_h
        return clo, top

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    # launch shape: empirical tuner (cached per graph class), untimed
    if args.shape:
        parts = args.shape.split(",")
        shape = {"walkers": int(parts[0]), "regs": int(parts[1]),
                 "order": parts[2] if len(parts) > 2 else "auto", "fixed": True}
    else:
        shape_probe = fc.Graph(rowptr_d, colidx_d, None, [ALPHA])
        shape = tune.autotune(shape_probe, tau)
        shape_probe.close()
    for i in range(args.warmup):
        step(1000 + i)
    torch.cuda.synchronize()

    # ---- device-resident inputs ----
    clocks = ClockSampler(local)
    clocks.start()
    step_ms, samp_ms, stats = [], [], []
    launches0 = fc.launch_count()
    nvtx_push("timed")  # profilers can restrict a capture to this range
    for i in range(args.steps):
        flush.zero_()
        torch.cuda.synchronize()
        barrier()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        sa, sb = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        step(2000 + i, samp_ev=(sa, sb), stats=stats)
        b.record(stream)
        torch.cuda.synchronize()
        barrier()
        step_ms.append(a.elapsed_time(b))
        samp_ms.append(sa.elapsed_time(sb))
    nvtx_pop()
    launches = fc.launch_count() - launches0
    clk = clocks.stop()
    R_sum = int(R.sum().item())

    # ---- end to end through the public API with host buffers ----
    e2e_ms = []
    for i in range(0 if args.no_e2e else args.steps):
        flush.zero_()
        torch.cuda.synchronize()
        barrier()
        t0 = time.perf_counter()
        step(3000 + i, host_inputs=True)
        torch.cuda.synchronize()
        e2e_ms.append(1000.0 * (time.perf_counter() - t0))
        barrier()

    tot_ms = sum(step_ms)
    tot_e2e = sum(e2e_ms) if e2e_ms else float("nan")
    if world > 1:
        import torch.distributed as dist
        t = torch.tensor([tot_ms, tot_e2e], dtype=torch.float64, device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        tot_ms, tot_e2e = float(t[0]), float(t[1])
    ms_per_step = tot_ms / args.steps
    value = world * tau * args.steps / (tot_ms / 1000.0)
    e2e_value = world * tau * args.steps / (tot_e2e / 1000.0)

    # roofline of the dominant kernel (the persistent Wilson sampler):
    # algorithmic bytes = 20 B per walk step + 8 B per vertex and tree
    peaks, peak_kind = load_peaks()
    pops = statistics.mean(s_[0] for s_ in stats)
    deps = statistics.mean(s_[1] for s_ in stats)
    alg_bytes = algorithmic_bytes(deps, n, tau)
    # the walker kernels' own layout (not the cycle-popping kernel's)
    lay_bytes = None
    if launched.get("kernel") != 5:
        lay_bytes = layout_bytes(deps, pops, n, tau, R_sum if world == 1 else R_sum // world)
    samp_s = statistics.mean(samp_ms) / 1000.0
    achieved = alg_bytes / samp_s / 1e9
    peak = float(peaks.get("hbm_gbs", 6800.0))
    kname = {2: "k_wilson_edge<flags, {r}>", 3: "k_wilson_edge<smem bitmap, {r}>",
             4: "k_wilson_edge<global bitmap, {r}>", 5: "k_pop"}.get(
        launched.get("kernel"), "k_wilson<global state, {r}>").format(r=launched.get("regs"))
    traffic = profiled_traffic(kname, launched) if full else None
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                "frac": achieved / peak, "traffic": traffic,
                "traffic_over_algorithmic": (traffic / alg_bytes) if traffic else None,
                "algorithmic_bytes": alg_bytes,
                "algorithmic_bytes_rule": "20 B per walk step + 8 B per vertex and tree",
                "layout_bytes": lay_bytes, "layout_frac": lay_bytes / samp_s / 1e9 / peak if lay_bytes else None,
                "kernel": kname, "launch": launched,
                "peak_source": peak_kind, "kernel_ms": 1000.0 * samp_s,
                "departures_per_launch": deps, "pops_per_launch": pops,
                "steps_per_s": deps / samp_s,
                # DRAM bytes per walk step, from the committed capture's traffic
                "dram_bytes_per_departure": (traffic / deps) if traffic else None}

    # accuracy of the last step's estimate (untimed): diag(Omega) against CG
    # columns of the library's solver on degree-stratified reference vertices
    accuracy = None
    if rank == 0 and full and not args.no_e2e:
        J = reference_vertices(g, 256, 5)
        Gj = fc.Graph(rowptr_d, colidx_d, None, [ALPHA])
        B = torch.zeros(J.size, n, dtype=torch.float64, device=dev)
        Jt = torch.from_numpy(J).to(dev)
        B[torch.arange(J.size, device=dev), Jt] = 1.0
        X, _ = Gj.solve(B, rel_tol=1e-10)
        ref = X[torch.arange(J.size, device=dev), Jt]
        Gj.close()
        err = (last_diag[0][Jt] - ref).abs()
        accuracy = {"reference_vertices": int(J.size), "max_abs_err": float(err.max()),
                    "mean_abs_err": float(err.mean()),
                    "hoeffding_bound_delta_1e-6": math.sqrt(math.log(2e6) / (2 * world * tau))}
        del B, X
    del flush

    tte_graphs = None
    if tte_gen is not None:
        ex, futs = tte_gen
        tte_graphs = [f.result() for f in futs]
        ex.shutdown()

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, cores, total, dt = cpu_trees_per_s(g, trees_per_core=4)
        st_trees, st_steps = cpu_single_thread(g)
        cpu = {"value": rate, "unit": "trees/s", "cores": cores, "kind": "oracle",
               "sample": f"{total} trees of the workload ({dt:.1f} s wall), 4 per host core, "
                         f"sequential Wilson (Algorithm 2) per thread",
               "single_thread": {"trees_per_s": st_trees, "walk_steps_per_s": st_steps, "trees": 2}}

    tte = None
    if tte_graphs is not None:
        tte, _ = cv_study(tte_graphs[0], tte_graphs[1:], args.seeds, args.rmat_scale)

    if rank == 0:
        line = {
            "metric": "USTs/s", "value": value, "unit": "trees/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "u32/f64", "data": "synthetic",
            "config": bench_config(args, g, world),
            "sampler_shape": shape,
            "e2e": {"value": e2e_value, "unit": "trees/s", "h2d_bytes_per_step": 8 * (n + 1) + 4 * nnz,
                    "d2h_bytes_per_step": 8 * n + 4 * TOPK},
            "gpu_launches": int(launches),
            "roofline": roofline,
            "cpu_baseline": cpu,
            "clocks": clk,
            "sampling_ms_per_step": statistics.mean(samp_ms),
            "accuracy": accuracy,
            "time_to_eps": tte,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
