"""Time-to-solution benchmark of the hybrid LOBPCG -> RMM-DIIS eigensolver (one JSON line).

Workload (the hybrid-solver configuration): n = 2,000,000, ~400 nonzeros per full row on a
seeded 256 x 256 block pattern, half-stored (~4e8 stored nonzeros), FP32 values and vectors;
the lowest n_ev = 8 eigenpairs, block n_b = 16, LOBPCG front to relative residual 1e-2, then
Jacobi-preconditioned batched RMM-DIIS to 1e-6.  The initial guess is the zero-padded lowest
eigenvectors of the leading n/10 principal block (the smaller-model-space start of Sec. 3.1),
computed beforehand on the GPU (FP64 LOBPCG to 1e-8) and excluded from the timing, as in the paper.

A step is one complete solve (eig_solve) with H resident in HBM.  The line also carries:
  * roofline / roofline_by_shape: the SpMM launches of the timed solves, per product shape
    (CUDA events on the solve's stream), against the measured HBM copy rate;
  * solve: iteration counts (including the LOBPCG safety net's, iterations_fallback), and the
    FP64 oracle's true residuals of the returned pairs with the eigenvalue error bound they give;
  * fp64_baseline: the same solve with FP64 values and vectors (the plain FP64 GPU solver);
  * e2e: the metric through the C ABI from host buffers (eig_create with H copied in and
    planned, eig_solve with a host X0, eig_ritz copying the eigenvectors back);
  * cpu_baseline: the FP64 oracle's hybrid solved on a smaller instance of the same workload
    (same generator, density, block pattern and seed at n/40 rows) on all host cores, scaled by
    stored nonzeros (oracle_sample; --impl reference times the same).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--n N] ...
  python bench.py --workload learned | batch | scale | sweep   (the other workloads)
N > 1 runs under torchrun: every rank solves its own replica (replicas only: the solve has no
data-parallel exchange on one node here), timing is max over ranks.
"""
import argparse
import dataclasses
import json
import os
import platform
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "time-to-solution, lowest n_ev eigenpairs at rel. residual 1e-6; SpMM HBM GB/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", "--rows", dest="n", type=int, default=2_000_000,
                    help="matrix dimension (--rows: the spelling to use under torchrun, whose own options "
                         "--nnodes / --nproc-per-node make --n ambiguous)")
    ap.add_argument("--nnz-per-row", type=float, default=400)
    ap.add_argument("--block-pattern", type=int, default=256)
    ap.add_argument("--nev", type=int, default=8)
    ap.add_argument("--nb", type=int, default=16)
    ap.add_argument("--tol", type=float, default=1e-6)
    ap.add_argument("--seed", type=int, default=1)
    ap.add_argument("--vec", default="f32", choices=["f32", "f64"])
    ap.add_argument("--storage", default="f32", choices=["f32", "f64", "bf16"])
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--rmm-precond", type=int, default=1, choices=[0, 1],
                    help="Jacobi-preconditioned RMM-DIIS corrections after the switch")
    ap.add_argument("--switch-res", type=float, default=1e-2,
                    help="switch to RMM-DIIS once every wanted relative residual is below this")
    ap.add_argument("--switch-tau", type=float, default=0.0,
                    help="switch on the eigenvalue-change rule tau <= this (0: off)")
    ap.add_argument("--switch-gap", type=float, default=0.03,
                    help="also wait until every wanted ||r_j|| <= this x the gap to the nearest other Ritz "
                         "value (0: off; not in the paper)")
    ap.add_argument("--s-max", type=int, default=10,
                    help="largest DIIS window of RMM-DIIS (Alg. 4 input s)")
    ap.add_argument("--layout", default="auto", choices=["auto", "mirrored", "half", "csr"],
                    help="device layout of the SpMM plan")
    ap.add_argument("--oracle-rows", type=int, default=0,
                    help="rows of the leading principal block the CPU oracle solves as its bounded sample "
                         "(0: n / 40)")
    ap.add_argument("--no-fp64-arm", action="store_true",
                    help="skip the FP64 values/vectors GPU arm of the hybrid line")
    ap.add_argument("--batch-count", type=int, default=32)
    ap.add_argument("--batch-threads", type=int, default=16)
    ap.add_argument("--workload", default="hybrid", choices=["hybrid", "learned", "batch", "scale", "sweep"],
                    help="hybrid: the time-to-solution line; learned: train the learned K on a matrix "
                         "family and compare it with Jacobi on held-out members; batch: 32 uneven "
                         "instances; scale: n = 8M, ~500 nnz/row with FP32 and BF16 values; sweep: the "
                         "switch-point sweep of Sec. 4 on a paper-shaped matrix")
    ap.add_argument("--scale-n", type=int, default=8_000_000)
    ap.add_argument("--scale-nnz-per-row", type=float, default=500)
    ap.add_argument("--scale-nev", type=int, default=10)
    ap.add_argument("--sweep-n", type=int, default=197_822)
    ap.add_argument("--sweep-nnz-per-row", type=float, default=1080)
    ap.add_argument("--sweep-max-switch", type=int, default=30)
    ap.add_argument("--lp-n", type=int, default=1_000_000)
    ap.add_argument("--lp-nnz-per-row", type=float, default=300)
    ap.add_argument("--lp-train", type=int, default=48)
    ap.add_argument("--lp-held", type=int, default=16)
    ap.add_argument("--lp-epochs", type=int, default=10)
    ap.add_argument("--lp-switch-res", type=float, default=1e-3,
                    help="learned workload: LOBPCG front to this residual, then RMM-DIIS (the family's "
                         "near-degenerate shells need a later switch than 1e-2)")
    return ap.parse_args()


def dist_setup(args):
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if ws > 1:
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        dist.init_process_group(backend)
    return ws, rank, local


def reduce_max(value, ws, device=None):
    if ws <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def barrier(ws):
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled every 200 ms during the timed region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu):
        self.gpu = gpu
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in self.lines:
            p = [x.strip() for x in l.split(",")]
            if len(p) < 9:
                continue
            try:
                sm.append(float(p[1]))
                mx = float(p[2])
            except ValueError:
                continue
            for nm, v in zip(names, p[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def measured_peak():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def make_problem(args):
    from gen import ci_matrix
    t = time.time()
    H = ci_matrix(args.n, args.nnz_per_row, args.block_pattern, seed=args.seed, storage=args.storage)
    return H, time.time() - t


def pinned(a, keep):
    """A copy of numpy array a in page-locked host memory (a numpy view of a pinned torch
    buffer, which `keep` holds alive)."""
    import torch
    a = np.ascontiguousarray(a)
    buf = torch.empty(a.nbytes, dtype=torch.uint8, pin_memory=True)
    keep.append(buf)
    v = buf.numpy().view(a.dtype).reshape(a.shape)
    v[...] = a
    return v


def initial_guess(H, args, binding):
    """Zero-padded lowest n_b eigenvectors of the leading n/10 principal block (the smaller model
    space of Sec. 3.1), solved on the GPU by LOBPCG with FP64 vectors to relative residual 1e-8,
    itself started from the padded eigenvectors of its own leading block of at most 20,000 rows
    (LOBPCG from a seeded random block).  A random block straight on n/10 rows can leave the
    shifted Jacobi preconditioner on an interior cluster of these spectra, whose lowest pairs are
    localised in the first rows."""
    from gen import principal_submatrix, pad_rows
    n0 = max(args.nb * 8, H.n // 10)
    n00 = max(args.nb * 8, min(20000, n0 // 10))
    X = None
    for m in (n00, n0):
        S0 = binding.Solver(principal_submatrix(H, m), args.nb, args.nb)
        if X is None:
            S0.solve("lobpcg", vec_type="f64", tol=1e-8, maxiter=1000, seed=args.seed)
        else:
            S0.solve("lobpcg", X0=pad_rows(X, m), vec_type="f64", tol=1e-8, maxiter=1000)
        X = S0.ritz()[1]
        S0.close()
    return pad_rows(X, H.n)


def oracle_sample(H, args, threads):
    """The CPU baseline, one model for both CPU legs: the FP64 oracle's hybrid (LOBPCG of Alg. 2,
    switched to RMM-DIIS of Alg. 4 by the bench's rule, Jacobi K) solved to the bench tolerance
    on a smaller instance of the same workload: the same generator, density, block pattern and
    seed at n_s rows (a bounded sample), from its own small-space start (lowest n_b eigenvectors
    of its leading n_s/10 block, oracle LOBPCG to 1e-8; not timed), as the GPU solve starts.  (A
    leading principal block of the bench matrix would not do: it keeps only the couplings of
    the low rows that fall inside it, a few percent of them, and converges at once.)  The
    oracle's products run on `threads` host threads (oracle.parallel_upper: row ranges, bitwise
    the single-threaded product).  Returns the measured seconds of the solve, the result and
    the sample matrix."""
    import oracle as O
    from gen import ci_matrix, principal_submatrix, pad_rows
    ns = args.oracle_rows or max(args.nb * 16, H.n // 40)
    Hs = ci_matrix(ns, args.nnz_per_row, args.block_pattern, seed=args.seed, storage=args.storage)
    n00 = max(args.nb * 4, ns // 10)
    Z00 = O.lobpcg(principal_submatrix(Hs, n00), np.random.default_rng(1).standard_normal((n00, args.nb)),
                   args.nb, tol=1e-8, maxiter=300).X
    Us = O.parallel_upper(Hs, threads)
    X0 = pad_rows(Z00, ns)
    t = time.perf_counter()
    r = O.hybrid(Hs, X0, args.nev, tol=args.tol, U=Us, rmm_maxiter=300,
                 rmm_precond="jacobi" if args.rmm_precond else "none",
                 switch_res=args.switch_res if args.switch_res > 0 else None,
                 switch_tau_tol=args.switch_tau if args.switch_tau > 0 else None, s_max=args.s_max,
                 switch_gap=args.switch_gap if args.switch_gap > 0 else None)
    dt = time.perf_counter() - t
    Us.pool.shutdown()
    return dt, r, Hs


def oracle_sample_desc(H, Hs, dt, r, threads):
    rm = r.extra["rmm"]
    return (f"FP64 oracle hybrid solved to the bench tolerance on the same generator at n = {Hs.n:,} "
            f"({Hs.nnz:,} stored nonzeros; {r.extra['front'].iterations} LOBPCG + "
            f"{rm.iterations if rm else 0} RMM-DIIS iterations, converged={bool(r.converged)}) in {dt:.2f} s on "
            f"{threads} host threads, scaled by stored nonzeros ({H.nnz:,} / {Hs.nnz:,}) to the bench matrix")


def cpu_baseline(H, args):
    threads = os.cpu_count() or 1
    dt, r, Hs = oracle_sample(H, args, threads)
    return {"value": dt * H.nnz / Hs.nnz * 1e3, "unit": "ms", "cores": threads, "kind": "oracle",
            "sample": oracle_sample_desc(H, Hs, dt, r, threads), "sample_s": dt}


def run_reference(args, ws, rank):
    """--impl reference: the FP64 CPU oracle on this workload (the paper's method has no
    published implementation to run, so the reference arm is the oracle).  Each step is one measured oracle_sample solve (ms_per_step is its wall time);
    `value` scales the median step to the bench matrix by stored nonzeros, as cpu_baseline does."""
    if rank != 0:
        return
    H, tgen = make_problem(args)
    threads = os.cpu_count() or 1
    times = []
    last = None
    for i in range(args.warmup + args.steps):
        dt, r, Hs = oracle_sample(H, args, threads)
        last = (dt, r, Hs)
        if i >= args.warmup:
            times.append(dt)
    med = statistics.median(times)
    step_ms = float(np.mean(times)) * 1e3
    value = med * H.nnz / last[2].nnz * 1e3
    desc = oracle_sample_desc(H, last[2], med, last[1], threads)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "ms", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": step_ms, "higher_is_better": False,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(args, H),
            "cpu_baseline": {"value": value, "unit": "ms", "cores": threads, "kind": "oracle",
                             "sample": f"median step: {desc}"},
            "e2e": {"value": value, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


SPMM_KERNELS = {1: "k_spmm_mirror (mirrored tiles, gather only)",
                2: "k_spmm_tiled + k_spmm_transpose_reduce (half-stored tiles)",
                3: "k_spmm_rowblock + k_spmm_transpose_reduce (CSR)"}


VAL_BYTES = {"f64": 8, "f32": 4, "bf16": 2}


def workload_config(args, H):
    rmm = "Jacobi-preconditioned RMM-DIIS" if args.rmm_precond else "RMM-DIIS"
    sw = []
    if args.switch_res > 0:
        sw.append(f"residual {args.switch_res:g}")
    if args.switch_tau > 0:
        sw.append(f"tau {args.switch_tau:g}")
    if getattr(args, "switch_gap", 0) > 0:
        sw = [" or ".join(sw) + f" and every wanted ||r|| <= {args.switch_gap:g} x gap"]
    return {"workload": (f"hybrid LOBPCG (to {' or '.join(sw)}) -> {rmm}, n={H.n:,}, ~{args.nnz_per_row:g} nnz/row, "
                         f"block pattern {args.block_pattern}, half-stored nnz={H.nnz:,}, "
                         f"{args.storage} values / {args.vec} vectors, n_ev={args.nev}, block {args.nb}, "
                         f"tol {args.tol:g}"),
            "n": H.n, "nnz_half": H.nnz, "n_ev": args.nev, "block": args.nb, "values": args.storage,
            "vectors": args.vec, "layout": args.layout, "switch_res": args.switch_res,
            "switch_tau": args.switch_tau, "switch_gap": getattr(args, "switch_gap", 0.0), "s_max": args.s_max,
            "l2": (f"inputs larger than L2 (stored matrix ~{(8 * (H.n + 1) + H.nnz * (4 + VAL_BYTES[args.storage])) / 1e9:.1f}"
                   " GB), no flush"),
            "parallelism": "replicas" if args.gpus > 1 else "single GPU"}


def run_learned(args, ws, rank, local):
    """The learned-preconditioner workload: H(g) = H0 + g V (n = --lp-n, ~--lp-nnz-per-row nonzeros
    per full row, block pattern 256, FP32 values; V on H0's pattern, N(0, 0.1^2)), g uniform in
    [0.5, 1.5].  The K is trained on LOBPCG iterates of the training members (on the GPU, by the
    library's kernels), then the hybrid solve (FP32 vectors, n_ev, block, tol 1e-6) with the
    learned K is timed against the same solve with the Jacobi K on each held-out member, from the
    small-space start.  Every rank runs the whole workload (replicas)."""
    import torch
    torch.cuda.set_device(local)
    from paper_2305_15552_gb300 import binding, learned as LG
    from gen import ci_matrix, family_perturbation, family_member
    lib = binding.load()
    t = time.time()
    H0 = ci_matrix(args.lp_n, args.lp_nnz_per_row, args.block_pattern, seed=args.seed, storage=args.storage)
    V = family_perturbation(H0, seed=args.seed + 100)
    tgen = time.time() - t
    gs = np.random.default_rng(args.seed).uniform(0.5, 1.5, args.lp_train + args.lp_held)
    samples, held_samples, held = [], [], []
    t = time.time()
    for q, g in enumerate(gs):
        Hq = family_member(H0, V, g)
        try:
            X0 = initial_guess(Hq, args, binding)
        except binding.EigError as e:   # a start that the small solve could not use: another seed
            print(f"member {q}: initial guess failed ({e}); retrying with another seed", file=sys.stderr)
            X0 = initial_guess(Hq, argparse.Namespace(**{**vars(args), "seed": args.seed + 17}), binding)
        S = binding.Solver(Hq, args.nev, args.nb)
        if q < args.lp_train:
            samples += LG.collect_samples(S, X0, iters=(0, 1, 2, 3, 5))
        else:
            held_samples += LG.collect_samples(S, X0, iters=(0, 2))
            held.append((g, X0))
        S.close()
    t_samples = time.time() - t
    p0 = LG.init_params(*LG.feature_stats(samples), seed=0)
    torch.cuda.synchronize()
    t = time.time()
    p, hist = LG.train(samples, p0, epochs=args.lp_epochs, lr=1e-3)
    torch.cuda.synchronize()
    t_train = time.time() - t
    loss_lp = LG.mean_loss(held_samples, p)
    loss_j = float(np.mean([LG.jacobi_loss(s_) for s_ in held_samples]))
    # throughput of the network kernel (inference on one sample's feature rows), FP32 ALU bound
    F = held_samples[0]["F"]
    for _ in range(3):
        binding.lp_forward(p, F)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    reps = 20
    with ClockSampler(local) as clk_mlp:
        e0.record()
        for _ in range(reps):
            binding.lp_forward(p, F)
        e1.record()
        torch.cuda.synchronize()
    mlp_ms = e0.elapsed_time(e1) / reps
    del samples, held_samples, F
    torch.cuda.empty_cache()
    # held-out solves: Jacobi K and learned K
    base = dict(vec_type=args.vec, tol=args.tol, timing=1, maxiter=500, switch_res=args.lp_switch_res,
                switch_tau=args.switch_tau, s_max=args.s_max)
    rows = []
    launches0 = lib.eig_launch_count()
    with ClockSampler(local) as clk:
        for g, X0 in held:
            Hq = family_member(H0, V, g)
            S = binding.Solver(Hq, args.nev, args.nb)
            X0d = torch.tensor(X0, device="cuda")
            res = {}
            for name, o in (("jacobi", dict(precond=1, rmm_precond=1)),
                            ("learned", dict(precond=2, rmm_precond=2, lp_params=p)),
                            ("learned_front", dict(precond=2, rmm_precond=1, lp_params=p)),
                            ("fp64_jacobi", dict(precond=1, rmm_precond=1, vec_type="f64"))):
                oo = {**base, **o}
                S.solve("hybrid", X0=X0d, **oo)        # warm-up
                torch.cuda.synchronize()
                e0.record()
                rc, st = S.solve("hybrid", X0=X0d, **oo)
                e1.record()
                torch.cuda.synchronize()
                res[name] = dict(ms=e0.elapsed_time(e1), rc=rc, front=st["iterations_front"],
                                 rmm=st["iterations_rmm"], safety=st["iterations_fallback"],
                                 spmm=st["spmm_calls"], lp_spmm=st["lp_spmm_calls"],
                                 k_fallback=st["precond_fallback"], max_relres=st["max_relres"])
            rows.append(res)
            S.close()
    launches = lib.eig_launch_count() - launches0
    ms_lp = float(np.mean([r["learned"]["ms"] for r in rows]))
    ms_j = float(np.mean([r["jacobi"]["ms"] for r in rows]))
    arms = ("jacobi", "learned", "learned_front", "fp64_jacobi")
    conv = {a: sum(r[a]["rc"] == 0 for r in rows) for a in arms}
    both = [r for r in rows if all(r[a]["rc"] == 0 for a in arms)]
    arm_ms = {a: float(np.mean([r[a]["ms"] for r in rows])) for a in arms}
    both_ms = {a: (float(np.mean([r[a]["ms"] for r in both])) if both else None) for a in arms}
    ms_val = reduce_max(arm_ms["learned_front"], ws, "cuda")
    clocks = clk.summary()
    props = torch.cuda.get_device_properties(local)
    mhz = clk_mlp.summary().get("sm_mhz") or clocks.get("sm_mhz") or 2070.0
    alu_peak = props.multi_processor_count * 128 * 2 * mhz * 1e6 / 1e12   # FP32 FMA lanes x 2 flops x clock
    flops_row = 2 * (6 * 32 + 32 * 32 + 32) + 20
    n_rows = args.lp_n * args.nev
    achieved = n_rows * flops_row / (mlp_ms * 1e-3) / 1e12
    line = {
        "metric": METRIC, "value": ms_val, "unit": "ms", "n_gpus": args.gpus, "steps": len(rows), "warmup": 1,
        "ms_per_step": ms_val, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": args.vec, "data": "synthetic",
        "config": {"workload": (f"learned preconditioner: H(g) = H0 + g V, n={args.lp_n:,}, ~{args.lp_nnz_per_row:g} "
                                f"nnz/row, block pattern {args.block_pattern}, {args.storage} values, g in [0.5, 1.5], "
                                f"{args.lp_train} training / {args.lp_held} held-out members; hybrid LOBPCG "
                                f"(to residual {args.lp_switch_res:g}) -> RMM-DIIS, n_ev={args.nev}, block {args.nb}, "
                                f"tol {args.tol:g}, learned K vs Jacobi K; value = mean held-out time-to-solution "
                                f"with the learned K in the LOBPCG front and Jacobi in RMM-DIIS (every arm in "
                                f"mean_ms: jacobi, learned in both phases, learned_front, fp64_jacobi = FP64 "
                                f"vectors with Jacobi)"),
                   "n": args.lp_n, "n_ev": args.nev, "block": args.nb, "train": args.lp_train,
                   "held_out": args.lp_held, "epochs": args.lp_epochs, "parallelism": "replicas" if ws > 1 else "single GPU",
                   "l2": "inputs larger than L2 (matrix ~1.2 GB), no flush"},
        "jacobi_ms": ms_j, "speedup_vs_jacobi": ms_j / arm_ms["learned_front"],
        "speedup_vs_fp64_jacobi": arm_ms["fp64_jacobi"] / arm_ms["learned_front"],
        "mean_ms": arm_ms,
        "converged": {**conv, "of": len(rows)},
        "all_converged": {"count": len(both), "mean_ms": both_ms},
        "held_out_loss": {"learned": loss_lp, "jacobi": loss_j},
        "per_matrix": rows,
        "gpu_launches": int(launches),
        "roofline": {"bound": "alu", "kernel": "k_lp_forward (6-32-32-1 MLP, FP32 FMA)", "achieved": achieved,
                     "peak": alu_peak, "unit": "TFLOP/s", "frac": achieved / alu_peak, "traffic": None,
                     "peak_kind": f"derived: {props.multi_processor_count} SMs x 128 FP32 lanes x 2 x {mhz:.0f} MHz",
                     "flops_per_row": flops_row, "rows_per_launch": n_rows, "avg_launch_ms": mlp_ms},
        "training": {"samples_s": t_samples, "train_s": t_train, "loss_first_epoch": hist[0],
                     "loss_last_epoch": hist[-1]},
        "clocks": clocks,
        "host": {"machine": platform.machine(), "cpus": os.cpu_count(), "gen_s": tgen},
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    barrier(ws)


def run_batch(args, ws, rank, local):
    """Batched uneven instances: --batch-count matrices with n log-uniform in [2e4, 5e5] and 50-300
    nonzeros per full row (same generator, block pattern 256, FP32 values, seed = base + index),
    n_ev = 5, block 8; each from its small-space start (computed beforehand, not timed).  Arms,
    each timed on the device over the whole batch: one instance after another on one stream;
    eig_solve_batch with worker streams; the same with each instance's SpMM plan shape chosen by
    eig_autotune_spmm (tuning not timed); lock-step (EIG_BATCH_LOCKSTEP, one thread per instance:
    each round's products of all running instances in one launch per shape).  Every rank runs the
    whole batch (replicas)."""
    import torch
    torch.cuda.set_device(local)
    from paper_2305_15552_gb300 import binding
    from gen import ci_matrix
    lib = binding.load()
    nev, nb = 5, 8
    a2 = argparse.Namespace(**{**vars(args), "nev": nev, "nb": nb})
    rng = np.random.default_rng(args.seed)
    ns = np.round(np.exp(rng.uniform(np.log(2e4), np.log(5e5), args.batch_count))).astype(int)
    nz = rng.uniform(50, 300, args.batch_count)
    t = time.time()
    Hs = [ci_matrix(int(n), float(z), args.block_pattern, seed=args.seed + 1000 + i, storage="f32")
          for i, (n, z) in enumerate(zip(ns, nz))]
    tgen = time.time() - t
    X0s = [torch.tensor(initial_guess(H, a2, binding), device="cuda") for H in Hs]
    opts = dict(vec_type="f32", tol=args.tol, maxiter=500, switch_res=args.lp_switch_res, switch_tau=0.0,
                s_max=args.s_max)
    tuned = [binding.autotune_spmm(H, nb, "f32", reps=3)[0] for H in Hs]
    S_def = [binding.Solver(H, nev, nb) for H in Hs]
    S_tun = [binding.Solver(H, nev, nb, layout=tb["layout"], row_block=tb["row_block"], col_block=tb["col_block"])
             for H, tb in zip(Hs, tuned)]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    res = {}

    def seq():
        out = []
        for S, X0 in zip(S_def, X0s):
            out.append(S.solve("hybrid", X0=X0, **opts))
        return out

    def timed(fn):
        fn()                                  # warm-up
        torch.cuda.synchronize()
        e0.record()
        out = fn()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1), out

    launches0 = lib.eig_launch_count()
    with ClockSampler(local) as clk:
        ms_seq, out_seq = timed(seq)
        ms_bat, out_bat = timed(lambda: binding.solve_batch(S_def, "hybrid", X0s=X0s, opts=opts,
                                                            threads=args.batch_threads))
        ms_tun, out_tun = timed(lambda: binding.solve_batch(S_tun, "hybrid", X0s=X0s, opts=opts,
                                                            threads=args.batch_threads))
        ms_lock, out_lock = timed(lambda: binding.solve_batch(S_def, "hybrid", X0s=X0s, opts=opts,
                                                              threads=args.batch_count, lockstep=True))
    lock_stats = out_lock[2][0]
    same_lock = all(sts_ == rc_ for sts_, (rc_, _) in zip(out_lock[1], out_seq))
    launches = lib.eig_launch_count() - launches0
    same = all(np.array_equal(a.ritz()[0], b.ritz()[0]) for a, b in zip(S_def, S_tun))
    conv_seq = sum(rc == 0 for rc, _ in out_seq)
    conv_bat = sum(s_ == 0 for s_ in out_bat[1])
    conv_tun = sum(s_ == 0 for s_ in out_tun[1])
    max_rel = max(float(np.max(S.ritz()[2])) for S in S_tun)
    for S in S_def + S_tun:
        S.close()
    ms_tun = reduce_max(ms_tun, ws, "cuda")
    layouts = {}
    for tb in tuned:
        k = f"{tb['layout']} {tb['row_block']}/{tb['col_block']}"
        layouts[k] = layouts.get(k, 0) + 1
    line = {
        "metric": METRIC, "value": ms_lock, "unit": "ms", "n_gpus": args.gpus, "steps": 1, "warmup": 1,
        "ms_per_step": ms_lock, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": (f"batched uneven instances: {args.batch_count} matrices, n log-uniform in "
                                f"[20,000, 500,000] (total {int(ns.sum()):,} rows), 50-300 nnz/row, block pattern "
                                f"{args.block_pattern}, FP32 values/vectors, n_ev={nev}, block {nb}, hybrid LOBPCG (to "
                                f"residual {args.lp_switch_res:g}) -> RMM-DIIS to {args.tol:g}; value = time to "
                                f"solve the whole batch in lock step (one SpMM launch per round over the running "
                                f"instances' row blocks, one thread and stream per instance)"),
                   "count": args.batch_count, "rows_total": int(ns.sum()), "n_ev": nev, "block": nb,
                   "threads": args.batch_threads, "parallelism": "replicas" if ws > 1 else "single GPU",
                   "l2": "inputs mostly smaller than L2 individually, ~6 GB in total; no flush"},
        "sequential_ms": ms_seq, "batched_ms": ms_bat, "batched_tuned_ms": ms_tun,
        "lockstep_ms": ms_lock,
        "lockstep": {"what": "eig_solve_batch_ex with EIG_BATCH_LOCKSTEP, one thread per instance: each "
                             "round's products of all running instances in one launch per shape over their "
                             "concatenated row blocks", "batched_launches": int(lock_stats["batch_launches"]),
                     "products_in_them": int(lock_stats["batch_products"]),
                     "converged": int(sum(s_ == 0 for s_ in out_lock[1])), "statuses_equal_sequential": bool(same_lock)},
        "speedup_vs_sequential": ms_seq / ms_lock, "instances_per_s": args.batch_count / (ms_lock * 1e-3),
        "converged": {"sequential": conv_seq, "batched": conv_bat, "batched_tuned": conv_tun,
                      "of": args.batch_count},
        "tuned_eigenvalues_equal_default": bool(same), "max_relres": max_rel, "tuned_shapes": layouts,
        "gpu_launches": int(launches), "clocks": clk.summary(),
        "host": {"machine": platform.machine(), "cpus": os.cpu_count(), "gen_s": tgen},
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    barrier(ws)


SHAPE_NAMES = {0: "FP32 vectors, nb 1", 1: "FP32 vectors, nb 2", 2: "FP32 vectors, nb 4", 3: "FP32 vectors, nb 8",
               4: "FP32 vectors, nb 16", 5: "FP32 vectors, nb 32", 6: "FP64 vectors, nb 1", 7: "FP64 vectors, nb 2",
               8: "FP64 vectors, nb 4", 9: "FP64 vectors, nb 8", 10: "FP64 vectors, nb 16",
               11: "FP64 vectors, nb 32"}

# DRAM bytes per layout entry of k_spmm_mirror, from one ncu capture per shape at n = 500,000
# (dram__bytes_read.sum + dram__bytes_write.sum over the plan's layout entries, 2.04e8); keyed
# by the shape index 6 * (FP64 vectors) + log2(nb); void once spmm_mirror.cu changes.
SPMM_TRAFFIC = {"kernel_sha": "2bd61e47e79eb4dd", "per_layout_entry": {4: 1.314712e9 / 204360448, 3: 1.266262e9 / 204360448,
                                                          9: 1.335377e9 / 204360448}}


def kernel_sha():
    import hashlib
    src = os.path.join(ROOT, "paper_2305_15552_gb300", "csrc", "spmm_mirror.cu")
    return hashlib.sha256(open(src, "rb").read()).hexdigest()[:16]


def spmm_traffic(shape, layout_entries):
    """Per-launch DRAM bytes of the mirrored kernel at this shape, or None when no capture of the
    current kernel source exists."""
    per = SPMM_TRAFFIC["per_layout_entry"].get(shape)
    if per is None or SPMM_TRAFFIC["kernel_sha"] != kernel_sha():
        return None
    return per * layout_entries


def roofline_entries(stats_sum, peak, peak_kind, pinfo):
    out = []
    for k in range(12):
        c = stats_sum["spmm_calls_by_shape"][k]
        if not c:
            continue
        ms = stats_sum["spmm_ms_by_shape"][k]
        by = stats_sum["spmm_bytes_by_shape"][k]
        ach = by / max(ms, 1e-12) / 1e6
        tr = spmm_traffic(k, pinfo["layout_entries"]) if pinfo["layout"] == 1 else None
        out.append({"shape": SHAPE_NAMES[k], "launches": int(c), "avg_launch_ms": ms / c,
                    "algorithmic_bytes_per_launch": by / c, "achieved": ach, "peak": peak, "unit": "GB/s",
                    "frac": ach / peak, "peak_kind": peak_kind, "traffic": tr,
                    "traffic_over_algorithmic": (tr / (by / c)) if tr else None})
    return out


def warm_solves(S, X0d, opts, warmup):
    import torch
    for _ in range(warmup):
        S.solve("hybrid", X0=X0d, **opts)
    torch.cuda.synchronize()


def timed_solves(S, X0d, opts, steps, st_):
    """steps solves between CUDA events on the solve's stream; per-shape SpMM stats summed over
    them."""
    import torch
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    acc = {"spmm_calls_by_shape": [0] * 12, "spmm_ms_by_shape": [0.0] * 12, "spmm_bytes_by_shape": [0.0] * 12,
           "time_ms_spmm": 0.0, "spmm_bytes": 0.0, "spmm_timed": 0}
    stats = rc = None
    ev0.record(st_)
    for _ in range(steps):
        rc, stats = S.solve("hybrid", X0=X0d, **opts)
        for k in ("spmm_calls_by_shape", "spmm_ms_by_shape", "spmm_bytes_by_shape"):
            acc[k] = [a + b for a, b in zip(acc[k], stats[k])]
        acc["time_ms_spmm"] += stats["time_ms_spmm"]
        acc["spmm_bytes"] += stats["spmm_bytes"]
        acc["spmm_timed"] += stats["spmm_timed"]
    ev1.record(st_)
    torch.cuda.synchronize()
    return ev0.elapsed_time(ev1) / steps, rc, stats, acc


def certify(H, th, X, threads):
    """The FP64 oracle's true relative residuals ||H z - z theta|| / |theta| of the returned pairs
    (one oracle product on the host threads), and the residual bound on the eigenvalue error:
    some eigenvalue lies within ||r_j|| of theta_j, i.e. |dlambda|/|lambda| <= ||r_j|| / (|theta_j| - ||r_j||)."""
    import oracle as O
    U = O.parallel_upper(H, threads)
    HX = O.sym_upper_matmul(H, X, U)
    U.pool.shutdown()
    R = HX - X * th[None, :]
    rn = np.linalg.norm(R, axis=0)
    rel = rn / np.abs(th)
    bound = rn / np.maximum(np.abs(th) - rn, 1e-300)
    return rel, bound


def run_hybrid(args, ws, rank, local):
    import torch
    torch.cuda.set_device(local)
    from paper_2305_15552_gb300 import binding
    lib = binding.load()
    H, tgen = make_problem(args)
    X0 = initial_guess(H, args, binding)
    X0d = torch.tensor(X0, device="cuda")
    S = binding.Solver(H, args.nev, args.nb, layout=args.layout)
    pinfo = S.spmm_info()
    opts = dict(vec_type=args.vec, tol=args.tol, timing=1, maxiter=500, rmm_precond=args.rmm_precond,
                switch_res=args.switch_res, switch_tau=args.switch_tau, switch_gap=args.switch_gap, s_max=args.s_max)
    st_ = torch.cuda.current_stream()
    warm_solves(S, X0d, opts, args.warmup)
    barrier(ws)
    torch.cuda.synchronize()
    launches0 = lib.eig_launch_count()
    with ClockSampler(local) as clk:
        torch.cuda.nvtx.range_push("timed")  # lets a profiler select the timed steps
        ms, rc, stats, acc = timed_solves(S, X0d, opts, args.steps, st_)
        torch.cuda.nvtx.range_pop()
    launches = lib.eig_launch_count() - launches0
    barrier(ws)
    ms = reduce_max(ms, ws, "cuda")
    th, X, rel = S.ritz()
    S.close()
    threads = os.cpu_count() or 1
    true_rel, dl_bound = certify(H, th, X, threads)
    # end to end through the C ABI from pinned host buffers: H and X0 copied in (and H planned),
    # the eigenvectors copied back, every step
    e2e_ms = []
    h2d = H.rowptr.nbytes + H.col.nbytes + H.val.nbytes + X0.nbytes
    d2h = H.n * args.nev * 8 + 2 * args.nev * 8
    keep = []
    Hp = dataclasses.replace(H, rowptr=pinned(H.rowptr, keep), col=pinned(H.col, keep), val=pinned(H.val, keep))
    X0p = pinned(X0, keep)
    Xout = pinned(np.zeros((H.n, args.nev)), keep)
    for _ in range(args.e2e_steps):
        torch.cuda.synchronize()
        t = time.perf_counter()
        torch.cuda.nvtx.range_push("e2e_create")
        S2 = binding.Solver(Hp, args.nev, args.nb, layout=args.layout)
        torch.cuda.nvtx.range_pop()
        S2.solve("hybrid", X0=X0p, vec_type=args.vec, tol=args.tol, maxiter=500, rmm_precond=args.rmm_precond,
                 switch_res=args.switch_res, switch_tau=args.switch_tau, switch_gap=args.switch_gap, s_max=args.s_max)
        S2.ritz(out=Xout)
        torch.cuda.synchronize()
        e2e_ms.append((time.perf_counter() - t) * 1e3)
        S2.close()
    del Hp, X0p, Xout, keep
    e2e = reduce_max(min(e2e_ms), ws, "cuda") if e2e_ms else None
    peak, peak_kind = measured_peak()
    achieved = (acc["spmm_bytes"] / max(acc["time_ms_spmm"], 1e-9)) / 1e6  # GB/s over every timed SpMM
    by_shape = roofline_entries(acc, peak, peak_kind, pinfo)
    dom = max(by_shape, key=lambda e: e["launches"] * e["avg_launch_ms"]) if by_shape else None
    line = {
        "metric": METRIC, "value": ms, "unit": "ms", "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": False,
        "scaling": "weak", "vs_baseline": None, "dtype": args.vec, "data": "synthetic",
        "config": workload_config(args, H),
        "e2e": {"value": e2e, "unit": "ms", "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)},
        "gpu_launches": int(launches),
        "roofline": {"bound": "hbm", "kernel": SPMM_KERNELS.get(pinfo["layout"], "symmetric SpMM"),
                     "scope": "every SpMM launch of the timed solves (shapes below)",
                     "layout_device_bytes": pinfo["device_bytes"], "layout_entries": pinfo["layout_entries"],
                     "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "peak_kind": peak_kind,
                     "traffic": (sum(e["traffic"] * e["launches"] for e in by_shape) / max(acc["spmm_timed"], 1)
                                 if by_shape and all(e["traffic"] for e in by_shape) else None),
                     "algorithmic_bytes_per_launch": acc["spmm_bytes"] / max(acc["spmm_timed"], 1),
                     "avg_launch_ms": acc["time_ms_spmm"] / max(acc["spmm_timed"], 1),
                     "launches_per_step": acc["spmm_timed"] / args.steps,
                     "dominant_shape": dom["shape"] if dom else None},
        "roofline_by_shape": by_shape,
        "solve": {"status": rc, "iterations_front": stats["iterations_front"],
                  "iterations_rmm": stats["iterations_rmm"], "iterations_fallback": stats["iterations_fallback"],
                  "spmv_count": stats["spmv_count"], "spmm_calls": stats["spmm_calls"],
                  "max_relres": stats["max_relres"], "switch_reason": stats["switch_reason"],
                  "spmm_share": acc["time_ms_spmm"] / (ms * args.steps),
                  "theta": [float(v) for v in th],
                  "oracle_true_relres_max": float(np.max(true_rel)),
                  "oracle_true_relres": [float(v) for v in true_rel],
                  "dlambda_rel_bound_max": float(np.max(dl_bound)),
                  "certified_by": ("the FP64 oracle's product H z on the host: max_j ||H z_j - z_j theta_j|| / "
                                   "|theta_j|; the eigenvalue error bound is the residual bound (some eigenvalue "
                                   "within ||r_j|| of theta_j)")},
        "clocks": clk.summary(),
        "host": {"machine": platform.machine(), "cpus": os.cpu_count(), "gen_s": tgen},
    }
    if not args.no_fp64_arm and args.vec == "f32" and args.storage == "f32":
        line["fp64_baseline"] = fp64_arm(args, binding, X0, line)
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(H, args)
    if rank == 0:
        print(json.dumps(line), flush=True)
    barrier(ws)


def fp64_arm(args, binding, X0, line):
    """The same hybrid solve with FP64 values and FP64 vectors throughout (the plain FP64 GPU solver
    the mixed-precision form is measured against): the same generator and seed with values kept in
    FP64, the same start, options and tolerance; one warm-up and two timed solves."""
    import torch
    from gen import ci_matrix
    torch.cuda.empty_cache()
    H64 = ci_matrix(args.n, args.nnz_per_row, args.block_pattern, seed=args.seed, storage="f64")
    S = binding.Solver(H64, args.nev, args.nb, layout=args.layout)
    opts = dict(vec_type="f64", tol=args.tol, timing=1, maxiter=500, rmm_precond=args.rmm_precond,
                switch_res=args.switch_res, switch_tau=args.switch_tau, switch_gap=args.switch_gap, s_max=args.s_max)
    X0d = torch.tensor(X0, device="cuda")
    warm_solves(S, X0d, opts, 1)
    ms, rc, stats, acc = timed_solves(S, X0d, opts, 2, torch.cuda.current_stream())
    th, X, _ = S.ritz()
    S.close()
    true_rel, _ = certify(H64, th, X, os.cpu_count() or 1)
    th32 = np.asarray(line["solve"]["theta"])
    return {"ms": ms, "status": rc, "iterations_front": stats["iterations_front"],
            "iterations_rmm": stats["iterations_rmm"], "iterations_fallback": stats["iterations_fallback"],
            "spmm_calls": stats["spmm_calls"], "spmm_ms_per_solve": acc["time_ms_spmm"] / 2,
            "oracle_true_relres_max": float(np.max(true_rel)),
            "speedup_fp32_over_fp64": ms / line["value"],
            "max_rel_diff_theta_vs_fp32": float(np.max(np.abs(th - th32) / np.abs(th))),
            "what": ("FP64 values and FP64 vectors through the same hybrid (LOBPCG -> RMM-DIIS), same start, "
                     "options and tolerance; one warm-up, mean of two timed solves")}


def run_scale(args, ws, rank, local):
    """Mixed precision at scale: n = --scale-n (8,000,000), ~--scale-nnz-per-row (500) nonzeros per
    full row, block pattern 256 (half-stored ~2.0e9 nonzeros, int64 rowptr, int32 columns), the
    lowest n_ev = --scale-nev (10) pairs, block 16, FP32 vectors; FP64 kept for the Grams, the
    projected problems and the DIIS solves.  Two arms: FP32 values and BF16 values (each the same
    generator and seed, values rounded to the storage type).  Each: small-space start (not timed),
    one warm-up and --steps timed solves of the hybrid (LOBPCG to residual 1e-2, then Jacobi-
    preconditioned RMM-DIIS to 1e-6), certified by the FP64 oracle's product on the host threads
    against that arm's own rounded H.  `value` is the FP32-values arm; precision_cost compares
    the BF16-values eigenvalues with the FP32-values ones."""
    import torch
    torch.cuda.set_device(local)
    from paper_2305_15552_gb300 import binding
    lib = binding.load()
    a2 = argparse.Namespace(**{**vars(args), "n": args.scale_n, "nnz_per_row": args.scale_nnz_per_row,
                               "nev": args.scale_nev, "nb": 16})
    peak, peak_kind = measured_peak()
    arms = {}
    launches = 0
    clocks = None
    for storage in ("f32", "bf16"):
        from gen import ci_matrix
        t = time.time()
        H = ci_matrix(a2.n, a2.nnz_per_row, a2.block_pattern, seed=a2.seed, storage=storage)
        tgen = time.time() - t
        X0 = initial_guess(H, a2, binding)
        X0d = torch.tensor(X0, device="cuda")
        S = binding.Solver(H, a2.nev, a2.nb, layout=args.layout)
        pinfo = S.spmm_info()
        opts = dict(vec_type="f32", tol=args.tol, timing=1, maxiter=500, rmm_precond=args.rmm_precond,
                    switch_res=args.switch_res, switch_tau=args.switch_tau, switch_gap=args.switch_gap,
                    s_max=args.s_max)
        warm_solves(S, X0d, opts, 1)
        l0 = lib.eig_launch_count()
        with ClockSampler(local) as clk:
            ms, rc, stats, acc = timed_solves(S, X0d, opts, args.steps, torch.cuda.current_stream())
        launches += lib.eig_launch_count() - l0
        if storage == "f32":
            clocks = clk.summary()
        th, X, _ = S.ritz()
        S.close()
        del X0d
        torch.cuda.empty_cache()
        true_rel, bound = certify(H, th, X, os.cpu_count() or 1)
        arms[storage] = {
            "ms": reduce_max(ms, ws, "cuda"), "status": rc, "nnz_half": H.nnz, "gen_s": tgen,
            "iterations_front": stats["iterations_front"], "iterations_rmm": stats["iterations_rmm"],
            "iterations_fallback": stats["iterations_fallback"], "spmm_calls": stats["spmm_calls"],
            "theta": [float(v) for v in th], "oracle_true_relres_max": float(np.max(true_rel)),
            "dlambda_rel_bound_max": float(np.max(bound)),
            "roofline_by_shape": roofline_entries(acc, peak, peak_kind, pinfo),
            "spmm_share": acc["time_ms_spmm"] / (ms * args.steps),
            "layout_device_bytes": pinfo["device_bytes"]}
        del H, X
    t32, t16 = np.asarray(arms["f32"]["theta"]), np.asarray(arms["bf16"]["theta"])
    r32 = arms["f32"]["roofline_by_shape"]
    dom = max(r32, key=lambda e: e["launches"] * e["avg_launch_ms"]) if r32 else None
    line = {
        "metric": METRIC, "value": arms["f32"]["ms"], "unit": "ms", "n_gpus": args.gpus, "steps": args.steps,
        "warmup": 1, "ms_per_step": arms["f32"]["ms"], "higher_is_better": False, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": (f"mixed precision at scale: n={a2.n:,}, ~{a2.nnz_per_row:g} nnz/row, block pattern "
                                f"{a2.block_pattern}, half-stored nnz={arms['f32']['nnz_half']:,}, FP32 values (value) "
                                f"and BF16 values (bf16 arm) with FP32 vectors, n_ev={a2.nev}, block 16, hybrid LOBPCG "
                                f"(to residual {args.switch_res:g}) -> Jacobi-preconditioned RMM-DIIS, tol {args.tol:g}"),
                   "n": a2.n, "n_ev": a2.nev, "block": 16, "parallelism": "replicas" if ws > 1 else "single GPU",
                   "l2": "inputs far larger than L2 (matrix ~16 GB), no flush"},
        "arms": arms,
        "precision_cost": {"max_rel_diff_theta_bf16_vs_f32": float(np.max(np.abs(t16 - t32) / np.abs(t32))),
                           "what": "eigenvalues of the BF16-rounded H against those of the FP32-rounded H, both "
                                   "certified to their own tolerance"},
        "roofline": dict(dom, bound="hbm", kernel=SPMM_KERNELS.get(1)) if dom else None,
        "gpu_launches": int(launches), "clocks": clocks,
        "host": {"machine": platform.machine(), "cpus": os.cpu_count()},
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    barrier(ws)


def run_sweep(args, ws, rank, local):
    """Switch-point sweep of the hybrid (Sec. 4, its fixed-switch tables and the optimal-vs-tau
    tables of Sec. 4.1) on a paper-shaped synthetic matrix: n = --sweep-n (197,822, the size of
    the 6Li N_max = 6 problem of Table 2), ~--sweep-nnz-per-row (1080) nonzeros per full row (the
    density of the paper's matrices), block pattern 256, FP32 values and FP64 vectors (the paper's
    precision).  For n_ev = 5
    (n_b = 8) and n_ev = 10 (n_b = 16), and for both fronts (LOBPCG, block Lanczos): the front
    alone to 1e-6, RMM-DIIS switched in after 5 / 10 / 15 / 20 front iterations, at tau <= 1e-4 and
    tau <= 1e-7 (Eq. switchtau), and every switch point 1..--sweep-max-switch, whose fewest SpMVs
    is the optimum.  RMM-DIIS runs as printed (unpreconditioned, no LOBPCG safety net); a run that
    does not converge within 500 iterations is reported unconverged.  SpMV counts as Sec. 2.6
    counts them; times are single solves between CUDA events after one warm-up per method.
    Also: block Lanczos alone with its thick restart (default), without restart and with a basis
    of 8 blocks; for n_ev = 5, decoupled RMM-DIIS (one SpMV per remaining vector once c = 1..4
    have converged, Sec. 4.3) against the coupled block product, with the time in products and
    its "effective SpMV" count (that time over the time of one SpMV).
    `value` is the LOBPCG -> RMM-DIIS hybrid at tau <= 1e-7, n_ev = 5."""
    import torch
    torch.cuda.set_device(local)
    from paper_2305_15552_gb300 import binding
    from gen import ci_matrix
    lib = binding.load()
    t = time.time()
    H = ci_matrix(args.sweep_n, args.sweep_nnz_per_row, args.block_pattern, seed=args.seed, storage="f32")
    tgen = time.time() - t
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    l0 = lib.eig_launch_count()
    tables = {}
    value = None
    with ClockSampler(local) as clk:
        for nev, nb in ((5, 8), (10, 16)):
            a2 = argparse.Namespace(**{**vars(args), "nev": nev, "nb": nb})
            X0 = torch.tensor(initial_guess(H, a2, binding), device="cuda")
            S = binding.Solver(H, nev, nb)
            base = dict(vec_type="f64", tol=args.tol, maxiter=500, rmm_maxiter=500, rmm_fallback=0, rmm_precond=0,
                        s_max=args.s_max, switch_res=0.0, timing=1)

            def run(method, **o):
                S.solve(method, X0=X0, **{**base, **o})
                torch.cuda.synchronize()
                e0.record()
                rc, st = S.solve(method, X0=X0, **{**base, **o})
                e1.record()
                torch.cuda.synchronize()
                k1 = 6                                   # FP64 vectors, block width 1 (SpMV launches)
                return {"converged": rc == 0, "spmv": int(st["spmv_count"]), "ms": e0.elapsed_time(e1),
                        "front_iterations": st["iterations_front"], "rmm_iterations": st["iterations_rmm"],
                        "products_ms": float(sum(st["spmm_ms_by_shape"])),
                        "spmv_launches": int(st["spmm_calls_by_shape"][k1]),
                        "spmv_ms": float(st["spmm_ms_by_shape"][k1]),
                        "block_launches": int(sum(st["spmm_calls_by_shape"]) - st["spmm_calls_by_shape"][k1])}

            rows = {}
            for front in ("lobpcg", "block_lanczos"):
                fr = {"alone": run(front, switch_tau=0.0)}
                for k in (5, 10, 15, 20):
                    fr[f"after_{k}"] = run("hybrid", front=front, switch_after=k, switch_tau=0.0)
                for tau in (1e-4, 1e-7):
                    fr[f"tau_{tau:g}"] = run("hybrid", front=front, switch_tau=tau)
                allk = [run("hybrid", front=front, switch_after=k, switch_tau=0.0)
                        for k in range(1, args.sweep_max_switch + 1)]
                conv = [(r["spmv"], k + 1, r) for k, r in enumerate(allk) if r["converged"]]
                if conv:
                    sp, kbest, rbest = min(conv, key=lambda z: (z[0], z[1]))
                    fr["optimum"] = dict(rbest, switch_after=kbest)
                fr["per_switch_point_spmv"] = [r["spmv"] if r["converged"] else None for r in allk]
                rows[front] = fr
            for m in ("lanczos", "chebfilter", "rmmdiis"):
                rows[m] = run(m)
            # block Lanczos (f3): thick restart (the default, half the basis kept) against the old
            # stop at the basis limit, and with a basis of only 8 blocks
            rows["block_lanczos_no_restart"] = run("block_lanczos", switch_tau=0.0, lanczos_keep=-1)
            rows["block_lanczos_basis8"] = dict(run("block_lanczos", switch_tau=0.0, lanczos_maxbasis=8 * nb),
                                                basis_vectors=8 * nb)
            if nev == 5:
                # decoupled RMM-DIIS (f2, Sec. 4.3): after c = 1..4 converged vectors, one SpMV per
                # remaining vector; c = 0 keeps the block product throughout.  "effective_spmv" is
                # the time in products over the time of one SpMV (the paper divides by the
                # SpMM/SpMV GFLOPS ratio instead)
                dec = {}
                for front in ("lobpcg", "block_lanczos"):
                    for k in (5, 10, 15, 20):
                        for cdec in range(5):
                            dec[f"{front}_after_{k}_c{cdec}"] = run("hybrid", front=front, switch_after=k,
                                                                    switch_tau=0.0, rmm_decouple=cdec)
                per = [r["spmv_ms"] / r["spmv_launches"] for r in dec.values() if r["spmv_launches"]]
                t1 = statistics.median(per) if per else None
                for r in dec.values():
                    r["effective_spmv"] = (r["products_ms"] / t1) if t1 else None
                rows["decoupled_rmmdiis"] = dec
                rows["spmv_ms"] = t1
            tables[f"nev{nev}_nb{nb}"] = rows
            if nev == 5:
                value = rows["lobpcg"]["tau_1e-07"]["ms"]
            S.close()
    launches = lib.eig_launch_count() - l0
    line = {
        "metric": METRIC, "value": value, "unit": "ms", "n_gpus": args.gpus, "steps": 1, "warmup": 1,
        "ms_per_step": value, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64", "data": "synthetic",
        "config": {"workload": (f"switch-point sweep (Sec. 4): paper-shaped n={H.n:,}, ~{args.sweep_nnz_per_row:g} "
                                f"nnz/row, block pattern {args.block_pattern}, half-stored nnz={H.nnz:,}, FP32 "
                                f"values, FP64 vectors (the paper's arithmetic for the vectors), Jacobi K in the front, "
                                f"unpreconditioned RMM-DIIS, tol {args.tol:g}, RMM-DIIS as printed (no safety net); value = "
                                f"LOBPCG -> RMM-DIIS at tau <= 1e-7, n_ev=5, n_b=8"),
                   "n": H.n, "parallelism": "replicas" if ws > 1 else "single GPU",
                   "l2": "matrix ~0.9 GB, larger than L2; no flush"},
        "tables": tables, "gpu_launches": int(launches), "clocks": clk.summary(),
        "host": {"machine": platform.machine(), "cpus": os.cpu_count(), "gen_s": tgen},
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    barrier(ws)


def main():
    args = parse()
    ws, rank, local = dist_setup(args)
    if args.workload == "batch" and args.impl == "ours":
        run_batch(args, ws, rank, local)
        return
    if args.workload == "learned" and args.impl == "ours":
        run_learned(args, ws, rank, local)
        return
    if args.workload == "scale" and args.impl == "ours":
        run_scale(args, ws, rank, local)
        return
    if args.workload == "sweep" and args.impl == "ours":
        run_sweep(args, ws, rank, local)
        return
    if args.impl == "reference":
        run_reference(args, ws, rank)
        barrier(ws)
        return
    run_hybrid(args, ws, rank, local)


if __name__ == "__main__":
    main()
