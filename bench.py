#!/usr/bin/env python
"""Benchmark: space-time predictor element-updates/s on one GB300.

Workload: the isolated-element population of the paper's performance proxy
(random tetrahedra, random data, one predictor per element): 200,000 seeded
tetrahedra, per-element Biot material, Q0 ~ N(0,1), degree N = 6.
One step = one predictor of every element (solve + time integration),
inputs resident in HBM.  Prints one JSON line (rank 0).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "predictor element-updates/s at N=6, FP64 vs mixed (≤1e-10 rel); served p50/p99"
UNIT = "element-updates/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--degree", type=int, default=6)
    ap.add_argument("--n-elem", type=int, default=200_000)
    ap.add_argument("--precision", default="both", choices=["both", "fp64", "mixed", "bf16x3"])
    ap.add_argument("--refine", type=int, default=1, choices=[0, 1, 2])
    ap.add_argument("--cpu-budget-s", type=float, default=12.0)
    ap.add_argument("--cpu-elems", type=int, default=16384,
                    help="elements of the workload the timed CPU baseline runs (repeated over the budget)")
    ap.add_argument("--ref-elems", type=int, default=4096, help="elements per step of the --impl reference arm")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-lu", action="store_true")
    ap.add_argument("--lu-n6", type=int, default=4, help="elements factored at N=6 for the LU comparator")
    ap.add_argument("--lu-n3", type=int, default=1024, help="elements factored at N=3 for the LU comparator")
    ap.add_argument("--no-steps", action="store_true", help="skip the time-stepping / LTS sections")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--no-sweeps", action="store_true", help="skip the degree and refinement sweeps")
    ap.add_argument("--sweep-degrees", type=int, nargs="*", default=[3, 4, 5])
    ap.add_argument("--no-systems", action="store_true", help="skip the damped Maxwell and viscoelastic predictors")
    ap.add_argument("--lts-nz", type=int, default=12,
                    help="layered graded mesh of the LTS vs GTS section: 2nz x 2nz x nz Kuhn boxes, 24 nz^3 tets "
                         "(12: 41,472)")
    ap.add_argument("--lts-full-nz", type=int, default=44,
                    help="configured-size LTS run (44: 2,044,416 tets; 0: skip)")
    ap.add_argument("--lts-full-fp64", action="store_true", help="also run the configured-size LTS in FP64")
    ap.add_argument("--planewave-study", action="store_true",
                    help="run the plane-wave convergence study instead of the benchmark")
    ap.add_argument("--planewave-degrees", type=int, nargs="*", default=[1, 2, 3, 4, 5, 6])
    ap.add_argument("--serving-requests", type=int, default=16)
    ap.add_argument("--serving-cycles", type=int, default=4, help="steps of the largest cluster per served request")
    ap.add_argument("--serving-no-fp64", action="store_true", help="skip the one-at-a-time FP64 baseline trace")
    return ap.parse_args()


def _workload(args):
    return {"workload": f"isolated space-time predictor, {args.n_elem} random tetrahedra "
                        f"(aspect <= 4, h 50-200 m), Biot material +-20%, Q0~N(0,1), N={args.degree}",
            "n_elem_per_gpu": args.n_elem, "degree": args.degree, "solver": "block back-substitution (Algorithm 3)",
            "l2": "inputs larger than L2 (Q0 and Qt streamed every step)"}


# ------------------------------------------------------------------ multi-rank
def max_over_ranks(x, world, device):
    """The largest x over all ranks (the slowest rank sets the job's time);
    x itself for one rank.  `device` is the rank's GPU under NCCL, "cpu"
    under gloo."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_rate(per_rank_units, world, seconds):
    """Whole-job throughput: every rank processes per_rank_units in the
    slowest rank's time."""
    return per_rank_units * world / seconds


def rank_seed(rank):
    """Each rank draws its own population (weak scaling, no shared data)."""
    from paper_2108_10565_gb300 import inputs
    return inputs.SEED_ISOLATED + rank


# ------------------------------------------------------------------ clocks
CLOCK_FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
                "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
                "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")


class ClockSampler:
    def __init__(self, device):
        self.path = tempfile.mktemp(suffix=".csv")
        self.proc = None
        try:
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={CLOCK_FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(device)], stdout=self.f,
                                         stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ------------------------------------------------------------------ cpu baseline
def _cpu_population(N, n, seed):
    """Operators A^{j*}, E* and Q0 of the first n elements of the workload,
    computed by the oracle (not timed)."""
    from oracle import geometry, predictor
    from paper_2108_10565_gb300 import inputs

    d = inputs.isolated_elements(n, N, seed=seed)
    As = np.empty((n, 3, 13, 13))
    Es = np.empty((n, 13, 13))
    for i in range(n):
        mat = inputs.material_dict(d["materials"][i])
        dt = geometry.cfl_dt(d["vertices"][i], mat, N)
        As[i], Es[i] = predictor.element_operators(d["vertices"][i], mat, dt)
    return As, Es, d["Q0"]


def cpu_alg3_rate(N, budget_s, threads, n_elem, seed=None):
    """Element-updates/s of the oracle's plain-loop C Algorithm 3 (binary64,
    OpenMP over elements, no BLAS) on the first n_elem elements of the
    workload, repeated until budget_s has passed.  Returns (rate, threads
    used, elements per pass, passes, seconds)."""
    from oracle import alg3_c
    from paper_2108_10565_gb300 import inputs

    As, Es, Q0 = _cpu_population(N, n_elem, inputs.SEED_ISOLATED if seed is None else seed)
    ref = alg3_c.reference_arrays(N)
    alg3_c.predict_alg3_c(N, As[:64], Es[:64], Q0[:64], threads, ref)  # warm-up (threads, pages)
    t0 = time.perf_counter()
    passes = 0
    while passes == 0 or time.perf_counter() - t0 < budget_s:
        alg3_c.predict_alg3_c(N, As, Es, Q0, threads, ref)
        passes += 1
    el = time.perf_counter() - t0
    used = threads if threads > 0 else alg3_c.default_threads()
    return n_elem * passes / el, used, n_elem, passes, el


def cpu_dense_lu_rate(args, budget_s, n_min=1):
    """The oracle's definition (dense equilibrated LU of Eq. stp-lineq,
    numpy/LAPACK float64) on the host cores, first elements of the workload."""
    from oracle import geometry, predictor
    from paper_2108_10565_gb300 import inputs

    k_max = 64
    d = inputs.isolated_elements(k_max, args.degree)
    t0 = time.perf_counter()
    done = 0
    while done < k_max and (done < n_min or time.perf_counter() - t0 < budget_s):
        mat = inputs.material_dict(d["materials"][done])
        dt = geometry.cfl_dt(d["vertices"][done], mat, args.degree)
        As, Es = predictor.element_operators(d["vertices"][done], mat, dt)
        predictor.predict_dense(args.degree, As, Es, d["Q0"][done])
        done += 1
    el = time.perf_counter() - t0
    try:
        from threadpoolctl import threadpool_info

        cores = max(int(i.get("num_threads", 1)) for i in threadpool_info()) if threadpool_info() else os.cpu_count()
    except Exception:
        cores = os.cpu_count()
    return done / el, cores, done, el


def cpu_other_systems(N, budget_s):
    """The oracle on the other systems' workloads (bounded samples, numpy):
    Algorithm 3 on damped-Maxwell and viscoelastic elements and the dense
    solve of the sub-cell material system, element-updates/s."""
    from oracle import maxwell, predictor, subcell, viscoelastic
    from paper_2108_10565_gb300 import inputs

    out = {}

    def timed(name, n, prep, solve):
        t0 = time.perf_counter()
        done = 0
        while done < n and (done == 0 or time.perf_counter() - t0 < budget_s):
            solve(*prep(done))
            done += 1
        el = time.perf_counter() - t0
        out[name] = {"element_updates_per_s": done / el, "sample": f"first {done} elements, {el:.1f} s"}

    dm = inputs.maxwell_isolated_elements(64, N)

    def prep_m(i):
        m = inputs.maxwell_dict(dm["materials"][i])
        As, Es = maxwell.element_operators(dm["vertices"][i], m, maxwell.cfl_dt(dm["vertices"][i], m, N))
        return As, Es, dm["Q0"][i]

    timed("damped_maxwell_alg3_numpy", 64, prep_m, lambda A, E, q: predictor.predict_alg3(N, A, E, q))
    dv = inputs.viscoelastic_isolated_elements(16, N)

    def prep_v(i):
        m = inputs.viscoelastic_dict(dv["materials"][i])
        As, Es = viscoelastic.element_operators(dv["vertices"][i], m, viscoelastic.cfl_dt(dv["vertices"][i], m, N))
        return As, Es, dv["Q0"][i]

    timed("viscoelastic_alg3_numpy", 16, prep_v, lambda A, E, q: predictor.predict_alg3(N, A, E, q))
    ds = inputs.subcell_isolated_elements(2, N, spread=0.1)

    def prep_s(i):
        from oracle import geometry
        mats = [inputs.material_dict(r) for r in ds["materials"][i]]
        dt = min(geometry.cfl_dt(ds["vertices"][i], m, N) for m in mats)
        As, Es = subcell.element_operators(ds["vertices"][i], mats, dt)
        return As, Es, ds["Q0"][i]

    timed("biot_subcell_dense_lu", 2, prep_s, lambda A, E, q: subcell.predict_dense(N, A, E, q))
    return out


def cpu_baseline(args):
    """The oracle timed on the host cores: the plain-loop C Algorithm 3 on all
    cores (the baseline), on one core, and the dense-LU definition; the
    oracle on the other systems' workloads beside them."""
    nall = args.cpu_elems
    rate, cores, k, passes, el = cpu_alg3_rate(args.degree, args.cpu_budget_s, 0, nall)
    r1, _, k1, p1, el1 = cpu_alg3_rate(args.degree, args.cpu_budget_s / 3, 1, max(64, nall // 16))
    lu, lu_cores, lu_k, lu_el = cpu_dense_lu_rate(args, args.cpu_budget_s / 3)
    other = None if args.no_systems else cpu_other_systems(args.degree, args.cpu_budget_s / 4)
    return {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle", "other_systems": other,
            "sample": f"oracle Algorithm 3 as plain C loops (binary64, OpenMP over elements, no BLAS, "
                      f"-ffp-contract=off): first {k} elements of the N={args.degree} workload, {passes} passes, "
                      f"{el:.1f} s on {cores} threads",
            "one_core": {"value": r1, "sample": f"first {k1} elements, {p1} passes, {el1:.1f} s"},
            "dense_lu_definition": {"value": lu, "cores": lu_cores,
                                    "sample": f"first {lu_k} elements, dense equilibrated LU (numpy/LAPACK), "
                                              f"{lu_el:.1f} s"}}


# ------------------------------------------------------------------ reference arm
def run_reference(args):
    """The oracle on the host cores: each step runs the plain-loop C
    Algorithm 3 (binary64, all cores) on a sample of the workload's
    elements (the first --ref-elems elements)."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from oracle import alg3_c
    from paper_2108_10565_gb300 import inputs

    N, n = args.degree, args.ref_elems
    As, Es, Q0 = _cpu_population(N, n, inputs.SEED_ISOLATED)
    ref = alg3_c.reference_arrays(N)
    for _ in range(args.warmup):
        alg3_c.predict_alg3_c(N, As, Es, Q0, 0, ref)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        alg3_c.predict_alg3_c(N, As, Es, Q0, 0, ref)
    el = time.perf_counter() - t0
    rate = n * args.steps / el
    cores = alg3_c.default_threads()
    sample = (f"{n} elements per step (the first {n} of the N={N} workload), oracle Algorithm 3 as plain C loops "
              f"(binary64, OpenMP over elements, no BLAS)")
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": _workload(args),
        "cpu_baseline": {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}))


# ------------------------------------------------------------------ our arm
# Issue cost of the double-binary32 kernel, in instruction slots of the 128-lane
# binary32 rate: a 32 x 32 + 64 bit integer multiply-add (measured at 13 to 19
# lanes a clock and SM, here 16) and a double-word multiply-add of 12 binary32
# instructions.
WIDE_MAC_SLOTS = 8.0
DW_OPS_PER_MAC = 12.0
# DRAM bytes (read + write) per element of the headline kernels at N = 6, from
# one ncu capture each of the 20,000-element case (dram__bytes_read.sum +
# dram__bytes_write.sum divided by the elements); the traffic grows in
# proportion to the elements, so a launch of n elements moves n times this
TRAFFIC_BYTES_PER_ELEMENT = {("mixed", 6, 1): 76378.0, ("fp64", 6, None): 76369.0}
# nominal tf32 : bf16 dense tensor ratio (1.1 : 2.25 PFLOP/s)
TF32_PER_BF16 = 1.1 / 2.25


def tc_tile_flops(N, bf16=False):
    """Tensor-core flops of one sweep's Khat products as issued: per degree
    block g and direction, 3 split products of M = 128 rows, N = rows l (o_g
    rounded up to 16), K = block columns (d_g rounded to 8 for tf32, 16 for
    bf16)."""
    tot = 0
    for g in range(1, N + 1):
        o, d = g * (g + 1) * (g + 2) // 6, (g + 1) * (g + 2) // 2
        npad = 16 if o <= 16 else (o + 15) // 16 * 16
        kpad = (d + 15) // 16 * 16 if bf16 else (d + 7) // 8 * 8
        tot += 3 * 3 * 2 * 128 * npad * kpad
    return tot


def direct_work(N):
    """Work of one element in the predictor kernel (Biot), in lane operations:
    `arith` multiplies and multiply-adds in the kernel's arithmetic (25 a
    direction, mode of degree >= 1 and time mode for the star products, 57 + 3 T
    a mode and time mode for the time solves, one per row that a degree block's
    Khat sums reach), and `int_macs` entries of the integer Khat rows."""
    B, T = (N + 1) * (N + 2) * (N + 3) // 6, N + 1
    nnz = {1: 4, 2: 29, 3: 119, 4: 364, 5: 924, 6: 2058}[N]
    rows = sum(-(-((g + 1) * (g + 2) // 2) // 21) * (g * (g + 1) * (g + 2) // 6) for g in range(1, N + 1))
    return {"arith": 75 * (B - 1) * T + (57 + 3 * T) * B * T + 13 * T * rows, "int_macs": 13 * T * nnz}


def fp32_alu_peak_tflops(sm_mhz):
    """binary32 FMA peak: 152 SMs x 128 lanes x 2 flop x clock."""
    return 152 * 128 * 2 * sm_mhz * 1e6 / 1e12


def fp64_alu_peak_tflops(sm_mhz):
    """binary64 FMA peak: nominal 1.25 TFLOP/s at 2070 MHz (152 SMs, 2 FMA
    lanes per SM per clock), scaled to the sampled clock."""
    return 1.25 * sm_mhz / 2070.0


def lu_comparator(L, torch, dev, local, args, hbm_gbs):
    """Block back-substitution vs the dense-LU comparator (factors
    precomputed; the paper's comparison of Table flop-count)."""
    from paper_2108_10565_gb300 import inputs

    out = {}
    for N, n in ((6, args.lu_n6), (3, args.lu_n3)):
        if n <= 0:
            continue
        d = inputs.isolated_elements(n, N, seed=inputs.SEED_ISOLATED + 17)
        dt = L.poro_cfl_dt(N, d["vertices"], d["materials"])
        ctx = L.poro_create(local, N, L.PORO_FP64)
        try:
            L.poro_set_isolated(ctx, d["vertices"], d["materials"], dt)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            L.poro_lu_factor(ctx, 0, n)
            t_fac = time.perf_counter() - t0
            q0 = torch.from_numpy(d["Q0"]).to(dev)
            B = q0.shape[2]
            qt = torch.empty((n, 13, B, N + 1), dtype=torch.float64, device=dev)
            st = torch.cuda.Stream(device=local)
            times = {}
            for name, solver in (("lu_solve", L.PORO_SOLVE_LU), ("block", L.PORO_SOLVE_BLOCK)):
                for _ in range(2):
                    L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), None, solver, st.cuda_stream)
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                reps = 3
                with torch.cuda.stream(st):
                    e0.record(st)
                    for _ in range(reps):
                        L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), None, solver, st.cuda_stream)
                    e1.record(st)
                torch.cuda.synchronize()
                times[name] = e0.elapsed_time(e1) / reps * 1e-3
            s_unk = 13 * B * (N + 1)
            ceiling = hbm_gbs * 1e9 / (8.0 * s_unk * s_unk)
            out[f"N{N}"] = {
                "elements": n, "unknowns": s_unk, "factor_bytes_per_element": 8 * s_unk * s_unk,
                "factor_s_per_element": t_fac / n,
                "lu_solve_elements_per_s": n / times["lu_solve"],
                "lu_solve_hbm_ceiling_elements_per_s": ceiling,
                "block_fp64_elements_per_s_same_batch": n / times["block"],
                "block_over_lu_solve": times["lu_solve"] / times["block"],
            }
        finally:
            L.poro_destroy(ctx)
    return out


def predictor_sweeps(L, torch, dev, local, args, head_pop):
    """The isolated population (200k elements) at the other configured
    degrees in the three forms, and refinement sweeps K = 0 and 2 of both
    mixed forms at the headline degree (K = 1 is the headline), with their
    error against the FP64 kernel: element-updates/s (CUDA events, mean of 5
    launches after 2 warm-ups)."""
    from paper_2108_10565_gb300 import inputs

    n = args.n_elem
    out = {"degrees": {}, "refinement_N6": {}}
    st = torch.cuda.Stream(device=local)

    def timed(ctx, q0, qt, io):
        for _ in range(2):
            L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK,
                               st.cuda_stream)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(st):
            e0.record(st)
            for _ in range(5):
                L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK,
                                   st.cuda_stream)
            e1.record(st)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / 5

    for N in sorted(set(args.sweep_degrees) | {args.degree}):
        d = head_pop if N == args.degree else inputs.isolated_elements(n, N)
        dt = L.poro_cfl_dt(N, d["vertices"], d["materials"])
        q0 = torch.from_numpy(d["Q0"]).to(dev)
        B, T = d["Q0"].shape[2], N + 1
        qt = torch.empty((n, 13, B, T), dtype=torch.float64, device=dev)
        io = torch.empty((n, 13, B), dtype=torch.float64, device=dev)
        ref = None
        row = {}
        settings = [("fp64", L.PORO_FP64, None)]
        if N == args.degree:
            settings += [(f"{nm}_K{k}", pr, k) for nm, pr in (("mixed_tf32", L.PORO_FP32_REFINE),
                                                            ("mixed_bf16x3", L.PORO_BF16X3_REFINE)) for k in (0, 2)]
        else:
            settings += [("mixed_tf32", L.PORO_FP32_REFINE, 1), ("mixed_bf16x3", L.PORO_BF16X3_REFINE, 1)]
        for name, prec, k in settings:
            ctx = L.poro_create(local, N, prec)
            try:
                if k is not None:
                    L.poro_set_refinement(ctx, k)
                L.poro_set_isolated(ctx, d["vertices"], d["materials"], dt)
                ms = timed(ctx, q0, qt, io)
            finally:
                L.poro_destroy(ctx)
            r = {"ms_per_launch": ms, "element_updates_per_s": n / (ms * 1e-3)}
            if prec == L.PORO_FP64:
                ref = qt.clone()
            elif ref is not None:
                e = (torch.linalg.vector_norm((qt - ref).reshape(n, -1), dim=1)
                     / torch.linalg.vector_norm(ref.reshape(n, -1), dim=1)).cpu().numpy()
                r["error_vs_fp64"] = {"median": float(np.median(e)), "max": float(e.max())}
            if N == args.degree:
                out["refinement_N6"][name] = r
            else:
                row[name] = r
        if N != args.degree:
            if not args.no_cpu:
                # the oracle's plain-loop C Algorithm 3 at this degree, all
                # host cores, on a bounded prefix of the population
                rate, cores, k, passes, el = cpu_alg3_rate(N, args.cpu_budget_s / 4, 0, args.cpu_elems // 2)
                row["cpu_alg3_oracle"] = {"element_updates_per_s": rate, "cores": cores,
                                          "sample": f"first {k} elements, {passes} passes, {el:.1f} s"}
            out["degrees"][str(N)] = row
        del q0, qt, io, ref
        torch.cuda.empty_cache()
    return out


def other_systems(L, torch, dev, local, args):
    """The binary64 Algorithm-3 kernel on the paper's other systems with an
    upper-triangular source matrix (Section "Other applications"): damped
    Maxwell (6 quantities, 200,000 elements) and viscoelastic attenuation
    (27 quantities, 50,000 elements), isolated tetrahedra of the headline
    geometry at the headline degree.  Element-updates/s (CUDA events, mean of
    5 launches after 2 warm-ups) and the FP64 pipe fraction against the
    nominal 1.25 TFLOP/s (flops from poro_flop_count).  Then the sub-cell
    material predictor (Section "Limitations") on 20,000 Biot elements."""
    from paper_2108_10565_gb300 import inputs

    N = args.degree
    out = {}
    st = torch.cuda.Stream(device=local)
    for name, system, n, gen, setter in (
            ("damped_maxwell", L.PORO_SYSTEM_MAXWELL, 200_000, inputs.maxwell_isolated_elements,
             L.poro_set_isolated_maxwell),
            ("viscoelastic_3mech", L.PORO_SYSTEM_VISCOELASTIC, 50_000, inputs.viscoelastic_isolated_elements,
             L.poro_set_isolated_viscoelastic)):
        d = gen(n, N)
        dt = L.poro_cfl_dt_system(system, N, d["vertices"], d["materials"])
        nq = d["Q0"].shape[1]
        q0 = torch.from_numpy(d["Q0"]).to(dev)
        qt = torch.empty((n, nq, d["Q0"].shape[2], N + 1), dtype=torch.float64, device=dev)
        io = torch.empty_like(q0)
        ctx = L.poro_create(local, N, L.PORO_FP64, system=system)
        try:
            setter(ctx, d["vertices"], d["materials"], dt)
            for _ in range(2):
                L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK,
                                   st.cuda_stream)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            with torch.cuda.stream(st):
                e0.record(st)
                for _ in range(5):
                    L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK,
                                       st.cuda_stream)
                e1.record(st)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1) / 5
            f = L.poro_flop_count(ctx, 0)[0]
        finally:
            L.poro_destroy(ctx)
        ach = f * n / (ms * 1e-3) / 1e12
        out[name] = {"elements": n, "quantities": nq, "ms_per_launch": ms, "element_updates_per_s": n / (ms * 1e-3),
                     "flops_per_element": f, "fp64_tflops": ach, "fp64_frac_nominal": ach / 1.25}
        del q0, qt, io
        torch.cuda.empty_cache()
    # sub-cell material (Section "Limitations"): Biot with linearly varying
    # Jacobians, 20,000 elements, vertex materials +-10 % around each element's
    # material; the Richardson iteration stops at a relative change of 1e-13
    n = 20_000
    d = inputs.subcell_isolated_elements(n, N, spread=0.1)
    dt = np.minimum.reduce([L.poro_cfl_dt(N, d["vertices"], np.ascontiguousarray(d["materials"][:, v, :]))
                            for v in range(4)])
    q0 = torch.from_numpy(d["Q0"]).to(dev)
    qt = torch.empty((n, 13, d["Q0"].shape[2], N + 1), dtype=torch.float64, device=dev)
    io = torch.empty_like(q0)
    ctx = L.poro_create(local, N, L.PORO_FP64)
    try:
        L.poro_set_isolated_subcell(ctx, d["vertices"], d["materials"], dt)
        for _ in range(2):
            L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK,
                               st.cuda_stream)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(st):
            e0.record(st)
            for _ in range(3):
                L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK,
                                   st.cuda_stream)
            e1.record(st)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / 3
        it = L.poro_get_subcell_iterations(ctx, 0, n)
    finally:
        L.poro_destroy(ctx)
    out["biot_subcell_linear_10pct"] = {
        "elements": n, "ms_per_launch": ms, "element_updates_per_s": n / (ms * 1e-3),
        "iterations": {"median": float(np.median(np.abs(it))), "max": int(np.abs(it).max()),
                       "unconverged": int((it <= 0).sum())}}
    del q0, qt, io
    torch.cuda.empty_cache()
    return out


def _setup_mesh_ctx(L, N, prec, mesh, mats, C, local=0, graphs=True):
    ctx = L.poro_create(local, N, prec)
    L.poro_set_mesh(ctx, mesh["vertices"], mesh["tets"], mesh["neighbors"], mesh["face_tag"])
    L.poro_set_materials(ctx, mats)
    dt, cl = L.poro_set_clusters(ctx, 0.5, C, n_elem=mesh["tets"].shape[0])
    L.poro_set_graphs(ctx, graphs)
    return ctx, dt, cl


def cfg2_mesh_steps(L, local, args):
    """The mixed predictor + corrector configuration at N = 5 and 6 on the
    isolated population's materials: a periodic Kuhn mesh of 196,608 tets
    (32^3 boxes) stands in for isolated elements with permutation neighbours
    (the library's corrector needs conforming faces); each element's 10
    material parameters are scaled by U[0.8, 1.2] (skeleton moduli tied) and
    Q0 ~ N(0, 1), seed 2108105652.  A GTS step is the predictor and the
    corrector of every element.  Element-updates/s over 3 steps after one
    warm-up step, and each mixed form's relative L2 error per element after
    one step against the FP64 form."""
    from paper_2108_10565_gb300 import inputs

    mesh = inputs.kuhn_box_mesh(32)
    ne = mesh["tets"].shape[0]
    rng = np.random.Generator(np.random.PCG64(inputs.SEED_CFG2))
    mats = inputs.perturbed_materials(rng, ne, tie_skeleton=True)
    out = {"n_elem": ne}
    for N in (5, 6):
        B = (N + 1) * (N + 2) * (N + 3) // 6
        q0 = np.random.Generator(np.random.PCG64(inputs.SEED_CFG2 + N)).standard_normal((ne, 13, B))
        ref = None
        row = {}
        for name, prec in (("fp64", L.PORO_FP64), ("mixed_bf16x3_K1", L.PORO_BF16X3_REFINE)):
            t0 = time.perf_counter()
            ctx, dt, _ = _setup_mesh_ctx(L, N, prec, mesh, mats, 1, local)
            setup = time.perf_counter() - t0
            try:
                L.poro_set_dofs(ctx, q0)
                L.poro_advance(ctx, 1.5 * dt)  # one step (and the warm-up)
                q1 = L.poro_get_dofs(ctx)
                t0 = time.perf_counter()
                L.poro_advance(ctx, 4.5 * dt)
                el = time.perf_counter() - t0
            finally:
                L.poro_destroy(ctx)
            r = {"ms_per_step": el / 3 * 1e3, "element_updates_per_s": ne * 3 / el, "host_setup_s": setup}
            if ref is None:
                ref = q1
            else:
                e = np.linalg.norm((q1 - ref).reshape(ne, -1), axis=1) / np.linalg.norm(ref.reshape(ne, -1), axis=1)
                r["error_vs_fp64_after_one_step"] = {"median": float(np.median(e)), "max": float(e.max())}
            row[name] = r
        out[f"N{N}"] = row
    return out


def time_stepping_sections(L, local, args):
    """Full ADER-DG steps (predictor + corrector + sources + receivers) under
    global and clustered local time stepping; wall-clock time to solution of
    poro_advance (synchronous)."""
    from paper_2108_10565_gb300 import inputs

    out = {}
    # the small periodic scenario: 384 tets, N = 2, 50 steps, graphs on / off
    sc = inputs.config0_scenario()
    r = {}
    for graphs in (True, False):
        ctx, dt, _ = _setup_mesh_ctx(L, sc["N"], 0, sc["mesh"], sc["materials"], 1, local, graphs)
        L.poro_add_point_source(ctx, sc["source"]["x"], sc["source"]["w"], sc["source"]["f0"], sc["source"]["t0"])
        for x in sc["receivers"]:
            L.poro_add_receiver(ctx, x)
        L.poro_advance(ctx, 5.5 * dt)  # warm-up (kernel attributes, graph capture path)
        t0 = time.perf_counter()
        L.poro_advance(ctx, (5 + sc["n_steps"] + 0.5) * dt)
        el = time.perf_counter() - t0
        L.poro_destroy(ctx)
        r["graphs" if graphs else "no_graphs"] = {"seconds": el, "steps": sc["n_steps"],
                                                  "element_updates_per_s": 384 * sc["n_steps"] / el}
    out["periodic_384_N2_50_steps"] = r
    # larger periodic GTS run: predictor + corrector throughput at N = 5
    mesh = inputs.kuhn_box_mesh(20)
    ne = mesh["tets"].shape[0]
    mats = np.tile(inputs.REFERENCE_MATERIAL, (ne, 1))
    r = {}
    for name, prec in (("fp64", 0), ("mixed", 1)):
        ctx, dt, _ = _setup_mesh_ctx(L, 5, prec, mesh, mats, 1, local)
        L.poro_set_dofs(ctx, np.random.default_rng(0).standard_normal((ne, 13, 56)))
        L.poro_advance(ctx, 1.5 * dt)
        nsteps = 6
        t0 = time.perf_counter()
        L.poro_advance(ctx, (1 + nsteps + 0.5) * dt)
        el = time.perf_counter() - t0
        L.poro_destroy(ctx)
        r[name] = {"seconds": el, "steps": nsteps, "element_updates_per_s": ne * nsteps / el}
    out[f"periodic_{ne}_N5_gts"] = r
    out["cfg2_periodic_mesh_N5_N6"] = cfg2_mesh_steps(L, local, args)
    # clustered LTS vs GTS on the layered graded mesh, same simulated time:
    # the configured 32x grading (3 populated clusters) and a 512x grading
    # that populates all 6; per-cluster GPU time of one cycle
    for grading in (32.0, 512.0):
        mesh, mats = inputs.layered_graded_mesh(args.lts_nz, grading=grading)
        ne = mesh["tets"].shape[0]
        r = {"n_elem": ne, "degree": 5, "grading": grading}
        for name, prec in (("fp64", 0), ("mixed", 1)):
            res = {}
            for C in (6, 1):
                ctx, dt, cl = _setup_mesh_ctx(L, 5, prec, mesh, mats, C, local)
                L.poro_add_point_source(ctx, np.array([0.0, 0.0, -1010.0]), inputs.EXPLOSIVE_WEIGHTS, 5.0, 0.25,
                                        1e12)
                L.poro_add_receiver(ctx, np.array([0.0, 0.0, -1.0]))
                t_sim = 32 * dt  # one step of the largest cluster of the LTS run
                L.poro_advance(ctx, t_sim * 1.0000001)  # warm-up cycle
                t0 = time.perf_counter()
                L.poro_advance(ctx, 2 * t_sim * 1.0000001)
                el = time.perf_counter() - t0
                hist = np.bincount(cl, minlength=C).tolist()
                upd = sum(n * 32 / 2 ** c for c, n in enumerate(hist))
                res["lts" if C > 1 else "gts"] = {"seconds": el, "element_updates": upd,
                                                  "element_updates_per_s": upd / el, "clusters": hist}
                if C > 1:
                    ms = L.poro_cluster_times(ctx, 3 * t_sim * 1.0000001, C)
                    res["lts"]["cluster_gpu_ms_per_cycle"] = ms.tolist()
                    res["lts"]["cluster_element_updates_per_cycle"] = [n * 32 / 2 ** c for c, n in enumerate(hist)]
                L.poro_destroy(ctx)
            res["lts_speedup_time_to_solution"] = res["gts"]["seconds"] / res["lts"]["seconds"]
            res["lts_work_fraction_of_gts"] = res["lts"]["element_updates"] / res["gts"]["element_updates"]
            r[name] = res
        out[f"layered_graded_{int(grading)}x_lts_vs_gts"] = r
    # the configured size: 88 x 88 x 44 boxes (2,044,416 tets), 32x grading,
    # clustered LTS, one warm-up and one timed cycle, per-cluster times
    if args.lts_full_nz > 0:
        mesh, mats = inputs.layered_graded_mesh(args.lts_full_nz, grading=32.0)
        ne = mesh["tets"].shape[0]
        r = {"n_elem": ne, "degree": 5, "grading": 32.0}
        for name, prec in (("mixed", 1), ("fp64", 0)):
            if name == "fp64" and not args.lts_full_fp64:
                continue
            t0 = time.perf_counter()
            ctx, dt, cl = _setup_mesh_ctx(L, 5, prec, mesh, mats, 6, local)
            setup_s = time.perf_counter() - t0
            L.poro_add_point_source(ctx, np.array([0.0, 0.0, -1010.0]), inputs.EXPLOSIVE_WEIGHTS, 5.0, 0.25, 1e12)
            for x in inputs.LOH_RECEIVERS:
                L.poro_add_receiver(ctx, x)
            t_sim = 32 * dt
            L.poro_advance(ctx, t_sim * 1.0000001)
            t0 = time.perf_counter()
            L.poro_advance(ctx, 2 * t_sim * 1.0000001)
            el = time.perf_counter() - t0
            ms = L.poro_cluster_times(ctx, 3 * t_sim * 1.0000001, 6)
            L.poro_destroy(ctx)
            hist = np.bincount(cl, minlength=6).tolist()
            upd = sum(n * 32 / 2 ** c for c, n in enumerate(hist))
            r[name] = {"seconds_per_cycle": el, "element_updates_per_cycle": upd, "element_updates_per_s": upd / el,
                       "clusters": hist, "cluster_gpu_ms_per_cycle": ms.tolist(), "host_setup_s": setup_s,
                       "gts_element_updates_same_time": ne * 32,
                       "lts_work_fraction_of_gts": upd / (ne * 32.0)}
        out["layered_graded_32x_full_size"] = r
    return out


def _serving_trace(L, args, n_req=None, size=(10_000, 500_000), cycles=None, seed_offset=0):
    """The served-ensemble requests: mesh sizes uniform in 10k-500k tets (Kuhn
    boxes of a 20 x 20 x 10 km domain, n_x = n_y = 2 n_z, free surface on
    top), degree uniform in {3, 4, 5, 6}, a 500 m layer over a half-space
    with each request's materials perturbed by +-20 % per parameter (the
    three skeleton moduli by one common factor), one
    explosive source at 1-5 km depth, 4 surface receivers, rate-2 clusters
    (at most 2), --serving-cycles steps of the largest cluster each (the
    configured 1 s of simulated time is cut)."""
    from paper_2108_10565_gb300 import inputs

    rng = np.random.Generator(np.random.PCG64(inputs.SEED_SERVING + seed_offset))
    meshes = {}
    reqs = []
    cycles = args.serving_cycles if cycles is None else cycles
    for i in range(args.serving_requests if n_req is None else n_req):
        n_target = int(rng.uniform(*size))
        key = max(1, int(round((n_target / 24.0) ** (1.0 / 3.0))))  # the mesh's n_z
        if key not in meshes:
            meshes[key] = inputs.uniform_box_mesh_for(n_target)
        mesh = meshes[key]
        ne = mesh["tets"].shape[0]
        N = int(rng.integers(3, 7))
        # the request's material: the layer over the half-space, each scaled by
        # one U[0.8, 1.2] draw per parameter for the whole request
        layer = inputs.perturbed_materials(rng, 1, base=inputs.LAYER_MATERIAL, tie_skeleton=True)[0]
        half = inputs.perturbed_materials(rng, 1, base=inputs.HALFSPACE_MATERIAL, tie_skeleton=True)[0]
        depth = -mesh["vertices"][mesh["tets"]].mean(axis=1)[:, 2]
        mats = np.ascontiguousarray(np.where((depth < 500.0)[:, None], layer[None, :], half[None, :]))
        src = dict(x=np.array([rng.uniform(5e3, 15e3), rng.uniform(5e3, 15e3), -rng.uniform(1e3, 5e3)]),
                   w=inputs.EXPLOSIVE_WEIGHTS.copy(), f0=2.0, t0=0.6, amplitude=1e12)
        rec = [np.array([x, y, -1.0]) for x, y in rng.uniform(2e3, 18e3, (4, 2))]
        reqs.append(dict(N=N, mesh=mesh, mats=mats, src=[src], rec=rec, ne=ne, C=2))
    for rq in reqs:
        dt = L.poro_cfl_dt(rq["N"], rq["mesh"]["vertices"][rq["mesh"]["tets"]], rq["mats"])
        dt_min = dt.min()
        cl = np.minimum(rq["C"] - 1, np.floor(np.log2(dt / dt_min) + 1e-12)).astype(int)
        rq["hist"] = np.bincount(cl, minlength=rq["C"])
        rq["t_end"] = cycles * dt_min * 2 ** (rq["C"] - 1) * 1.0000001
        rq["updates"] = cycles * sum(int(h) * 2 ** (rq["C"] - 1 - c) for c, h in enumerate(rq["hist"]))
    return reqs


def _serve(L, local, reqs, arrivals, prec, slots, batched):
    srv = L.poro_server_create(local, 200 << 30, slots)
    L.poro_server_set_batching(srv, batched)
    tickets, keep = [], []
    t0 = time.perf_counter()
    for rq, ta in zip(reqs, arrivals):
        now = time.perf_counter() - t0
        if ta > now:
            time.sleep(ta - now)
        sc, k = L.make_scenario(rq["N"], rq["mesh"], rq["mats"], rq["t_end"], precision=prec,
                                max_clusters=rq["C"], sources=rq["src"], receivers=rq["rec"])
        keep.append(k)
        tickets.append(L.poro_submit(srv, sc))
    states = [L.poro_wait(srv, t, 1_800_000) for t in tickets]
    wall = time.perf_counter() - t0
    lat = np.array([L.poro_request_times(srv, t)[2] for t in tickets])
    L.poro_server_destroy(srv)
    upd = sum(r["updates"] for r in reqs)
    return {"wall_s": wall, "done": int(sum(s == L.PORO_REQ_DONE for s in states)),
            "requests_per_s": len(reqs) / wall, "element_updates_per_s": upd / wall,
            "p50_time_to_seismogram_s": float(np.percentile(lat, 50)),
            "p99_time_to_seismogram_s": float(np.percentile(lat, 99))}


def serving_section(L, local, args):
    """Served ensemble: the configured request distribution (see
    _serving_trace) under continuous batching in the mixed bf16 form:
      - capacity: all requests submitted at once, batched and stream mode;
      - the Poisson trace (mean 2 requests/s), batched;
      - a Poisson trace at 0.8 x the measured batched capacity;
      - the baseline: the Poisson trace one request at a time in FP64."""
    from paper_2108_10565_gb300 import inputs

    reqs = _serving_trace(L, args)
    n_req = len(reqs)
    rng = np.random.Generator(np.random.PCG64(inputs.SEED_SERVING + 1))
    gaps = rng.exponential(1.0, n_req)
    at_once = np.zeros(n_req)
    out = {"requests": n_req, "own_cycles_per_request": args.serving_cycles, "max_clusters": 2,
           "mesh_elements": [int(r["ne"]) for r in reqs], "degrees": [int(r["N"]) for r in reqs],
           "element_updates_total": int(sum(r["updates"] for r in reqs))}
    bf = L.PORO_BF16X3_REFINE
    out["capacity_batched_mixed"] = _serve(L, local, reqs, at_once, bf, 16, True)
    out["capacity_streams_mixed"] = _serve(L, local, reqs, at_once, bf, 16, False)
    out["batched_over_streams"] = (out["capacity_batched_mixed"]["element_updates_per_s"]
                                   / out["capacity_streams_mixed"]["element_updates_per_s"])
    out["poisson_2_per_s_batched_mixed"] = _serve(L, local, reqs, np.cumsum(gaps / 2.0), bf, 16, True)
    lam = 0.8 * out["capacity_batched_mixed"]["requests_per_s"]
    out["arrival_rate_0p8_capacity_per_s"] = lam
    out["poisson_0p8_capacity_batched_mixed"] = _serve(L, local, reqs, np.cumsum(gaps / lam), bf, 16, True)
    if not args.serving_no_fp64:
        out["poisson_2_per_s_one_at_a_time_fp64"] = _serve(L, local, reqs, np.cumsum(gaps / 2.0), L.PORO_FP64, 1,
                                                           False)
    # many small requests (2k-20k tets, 16 steps each), all at once: the case
    # where runs sharing launches matters
    small = _serving_trace(L, args, n_req=48, size=(2_000, 20_000), cycles=16, seed_offset=2)
    z = np.zeros(len(small))
    out["small_requests"] = {"requests": len(small), "mesh_elements": [int(r["ne"]) for r in small],
                             "degrees": [int(r["N"]) for r in small],
                             "element_updates_total": int(sum(r["updates"] for r in small)),
                             "capacity_batched_mixed": _serve(L, local, small, z, bf, 48, True),
                             "capacity_streams_mixed": _serve(L, local, small, z, bf, 48, False)}
    sm = out["small_requests"]
    sm["batched_over_streams"] = (sm["capacity_batched_mixed"]["element_updates_per_s"]
                                  / sm["capacity_streams_mixed"]["element_updates_per_s"])
    # tiny requests (500-3k tets, 64 steps each), all at once: launches of a
    # few hundred CTAs, where one launch per degree group and tick pays most
    tiny = _serving_trace(L, args, n_req=64, size=(500, 3_000), cycles=64, seed_offset=3)
    z = np.zeros(len(tiny))
    out["tiny_requests"] = {"requests": len(tiny), "mesh_elements": [int(r["ne"]) for r in tiny],
                            "degrees": [int(r["N"]) for r in tiny],
                            "element_updates_total": int(sum(r["updates"] for r in tiny)),
                            "capacity_batched_mixed": _serve(L, local, tiny, z, bf, 64, True),
                            "capacity_streams_mixed": _serve(L, local, tiny, z, bf, 64, False)}
    tn = out["tiny_requests"]
    tn["batched_over_streams"] = (tn["capacity_batched_mixed"]["element_updates_per_s"]
                                  / tn["capacity_streams_mixed"]["element_updates_per_s"])
    return out


def run_ours(args):
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    from paper_2108_10565_gb300 import _lib as L
    from paper_2108_10565_gb300 import inputs

    N, n = args.degree, args.n_elem
    dev = f"cuda:{local}"
    peaks = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}  # fallback when no measured peaks are present
    peaks_src = "fallback (6.8 TB/s, 1.9 PFLOP/s bf16)"
    try:
        peaks.update(json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))))
        peaks_src = "MEASURED_PEAKS.json"
    except Exception:
        pass
    tensor_bf16_burst = float(peaks["bf16_tflops"])
    hbm_gbs = float(peaks["hbm_gbs"])
    d = inputs.isolated_elements(n, N, seed=rank_seed(rank))
    dt = L.poro_cfl_dt(N, d["vertices"], d["materials"])
    B, T = d["Q0"].shape[2], N + 1
    # pinned host buffers of the end-to-end leg, allocated before the large
    # device allocations of the timed forms
    hq = hi = None
    if not args.no_e2e:
        hq = torch.from_numpy(d["Q0"]).pin_memory()
        hi = torch.empty((n, 13, B), dtype=torch.float64).pin_memory()
    q0 = torch.from_numpy(d["Q0"]).to(dev)
    stream = torch.cuda.Stream(device=local)
    sh = stream.cuda_stream
    forms = {"fp64": (L.PORO_FP64, 0), "mixed": (L.PORO_FP32_REFINE, args.refine),
             "mixed_bf16x3": (L.PORO_BF16X3_REFINE, args.refine)}
    order = ["fp64", "mixed", "mixed_bf16x3"] if args.precision == "both" else [
        "mixed_bf16x3" if args.precision == "bf16x3" else args.precision]
    res, qts = {}, {}
    for name in order:
        prec, sweeps = forms[name]
        ctx = L.poro_create(local, N, prec)
        if prec != L.PORO_FP64:
            L.poro_set_refinement(ctx, sweeps)
        L.poro_set_isolated(ctx, d["vertices"], d["materials"], dt)
        qt = torch.empty((n, 13, B, T), dtype=torch.float64, device=dev)
        io = torch.empty((n, 13, B), dtype=torch.float64, device=dev)

        def step():
            L.poro_predict_dev(ctx, 0, n, q0.data_ptr(), qt.data_ptr(), io.data_ptr(), L.PORO_SOLVE_BLOCK, sh)

        for _ in range(args.warmup):
            step()
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
        sampler = ClockSampler(local)
        time.sleep(0.3)
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
        with torch.cuda.stream(stream):
            evs[0].record(stream)
            for k in range(args.steps):
                step()
                evs[k + 1].record(stream)
        torch.cuda.synchronize()
        clocks = sampler.stop()
        per = [evs[k].elapsed_time(evs[k + 1]) for k in range(args.steps)]
        ms = max_over_ranks(evs[0].elapsed_time(evs[-1]) / args.steps, world, dev)
        f = L.poro_flop_count(ctx, sweeps)
        res[name] = dict(ctx=ctx, ms=ms, per=per, clocks=clocks, flops=f, sweeps=sweeps, prec=prec)
        qts[name] = qt
    # accuracy of the mixed forms against the FP64 form on every element
    errs = {}
    for name in ("mixed", "mixed_bf16x3"):
        if "fp64" in qts and name in qts:
            a, b = qts[name], qts["fp64"]
            e = (torch.linalg.vector_norm((a - b).reshape(n, -1), dim=1)
                 / torch.linalg.vector_norm(b.reshape(n, -1), dim=1)).double().cpu().numpy()
            errs[name] = {"vs": "fp64 kernel (pinned to the oracle at 1e-12)", "median": float(np.median(e)),
                          "p99": float(np.quantile(e, 0.99)), "max": float(e.max())}
    del qts

    def roofline(name):
        """Roofline of one form's kernel against the measured peaks
        (MEASURED_PEAKS.json): HBM copy bandwidth and, for the unrefined
        form, dense bf16 tensor throughput (tf32 = bf16 x the nominal
        tf32 : bf16 ratio).  `frac` is the largest fraction over those roofs
        and `bound` names it; the binary64 kernel, which neither roof bounds,
        reports its FP64 pipe against the nominal unit count x the sampled
        clock.  `model` keeps the double-binary32 kernel's own issue-slot model
        apart from these."""
        r = res[name]
        mhz = (r["clocks"] or {}).get("sm_mhz") or 2070.0
        t = statistics.mean(r["per"]) * 1e-3
        Bm, Tm = (N + 1) * (N + 2) * (N + 3) // 6, N + 1
        # Q0 and the element's (Z - e I)^{-1}, 3 scalars and 15 star factors in; Qt, I out
        alg_bytes = 8.0 * (13 * Bm + Tm * Tm + 18 + 13 * Bm * Tm + 13 * Bm)
        hbm_ach = alg_bytes * n / t / 1e9
        terms = {"hbm": {"achieved": hbm_ach, "peak": hbm_gbs, "unit": "GB/s", "frac": hbm_ach / hbm_gbs,
                         "algorithmic_bytes_per_element": alg_bytes}}
        work = direct_work(N)
        if r["prec"] == L.PORO_FP64 or r["sweeps"] == 2:  # binary64 arithmetic, Khat sums in integers
            ach = 2.0 * work["arith"] * n / t / 1e12
            peak = fp64_alu_peak_tflops(mhz)
            tb = TRAFFIC_BYTES_PER_ELEMENT.get(("fp64", N, None))
            terms["fp64_pipe"] = {"achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak}
            return {"bound": "alu", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
                    "traffic": tb * n if tb else None, "kernel": f"stp_direct_kernel<{N},Bin64>",
                    "binary64_operations_per_element": work["arith"],
                    "integer_multiply_adds_per_element": 2 * work["int_macs"],
                    "algorithmic_flops_per_element": r["flops"][0], "terms": terms,
                    "peak_source": "binary64 FMA pipe, nominal (152 SM x 2 FMA/clk x 2 flop x 2.07 GHz = 1.25 "
                                   "TFLOP/s) scaled to the sampled clock; no measured FP64 peak exists; the Khat "
                                   "products are integer sums and not counted"}
        if r["sweeps"] == 1:  # double-binary32 on the binary32 and integer pipes
            b = terms["hbm"]
            slots = {"double_word": DW_OPS_PER_MAC * work["arith"], "integer": (WIDE_MAC_SLOTS + 1) * work["int_macs"]}
            t_alu = sum(slots.values()) * n / (152 * 128 * mhz * 1e6)
            tb = TRAFFIC_BYTES_PER_ELEMENT.get(("mixed", N, 1))
            return {"bound": "hbm", "achieved": b["achieved"], "peak": b["peak"], "unit": b["unit"], "frac": b["frac"],
                    "traffic": tb * n if tb else None, "kernel": f"stp_direct_kernel<{N},Bin32x2>",
                    "peak_source": peaks_src + " (hbm_gbs)", "terms": terms,
                    "model": {"frac": t_alu / t, "bound_times_ms": {"binary32_issue": 1e3 * t_alu},
                              "slots_per_element": slots,
                              "derivation": f"issue at 152 SM x 128 lanes x {mhz:.0f} MHz: {DW_OPS_PER_MAC:g} slots per "
                                            f"double-word operation, {WIDE_MAC_SLOTS:g} + 1 per entry of the integer "
                                            "Khat rows; the kernel's own instruction mix, not a hardware roof"}}
        # the unrefined form: one binary32 sweep with its Khat products on the
        # tensor cores, dense degree blocks (o_g rows x d_g columns, 13 T
        # right-hand columns, 3 directions), 3 split products (algorithmic); the
        # tiles as issued pad rows to 128 and columns to the MMA shape
        bf = r["prec"] == L.PORO_BF16X3_REFINE
        tc_alg = sum(3 * (g * (g + 1) * (g + 2) // 6) * ((g + 1) * (g + 2) // 2) * 13 * Tm * 2 * 3
                     for g in range(1, N + 1))
        tc_peak = tensor_bf16_burst * (1.0 if bf else TF32_PER_BF16)
        tc_ach = tc_alg * n / t / 1e12
        terms["tensor"] = {"achieved": tc_ach, "peak": tc_peak, "unit": "TFLOP/s", "frac": tc_ach / tc_peak,
                           "dtype": "bf16" if bf else "tf32",
                           "peak_source": "measured bf16 burst" + ("" if bf else f" x {TF32_PER_BF16:.3f}"),
                           "algorithmic_flops_per_element": tc_alg,
                           "issued_flops_per_element": tc_tile_flops(N, bf)}
        bound = max(("hbm", "tensor"), key=lambda k: terms[k]["frac"])
        b = terms[bound]
        return {"bound": bound, "achieved": b["achieved"], "peak": b["peak"], "unit": b["unit"], "frac": b["frac"],
                "traffic": None, "kernel": f"stp_mixed_kernel<{N}" + (",bf16>" if bf else ">"),
                "peak_source": peaks_src + " (" + ("hbm_gbs" if bound == "hbm" else "bf16_tflops burst") + ")",
                "terms": terms}

    # headline: the faster mixed form among those within 1e-10 of the FP64
    # kernel on every element (or when the FP64 form did not run); else FP64
    def _accurate(name):
        e = errs.get(name)
        return name in res and (e is None or e["max"] <= 1e-10)
    ok = [k for k in ("mixed", "mixed_bf16x3") if _accurate(k)]
    head = min(ok, key=lambda k: res[k]["ms"]) if ok else None
    head = head or ("fp64" if "fp64" in res else next(iter(res)))
    hr = res[head]
    value = job_rate(n, world, hr["ms"] * 1e-3)

    # end to end through the C ABI with host buffers (pinned), headline form
    e2e = None
    if not args.no_e2e:
        ctx = hr["ctx"]
        hq_np, hi_np = hq.numpy(), hi.numpy()
        # one library call per step: Q0 host -> device, predictor, I device ->
        # host, with the copies of each chunk overlapped with other chunks' kernels
        for _ in range(max(1, args.warmup)):
            L.poro_predict_host(ctx, hq_np, out=hi_np)
        if world > 1:
            dist.barrier()
        t0 = time.perf_counter()
        per = []
        for _ in range(args.steps):
            t1 = time.perf_counter()
            L.poro_predict_host(ctx, hq_np, out=hi_np)
            per.append(time.perf_counter() - t1)
        e2e_s = max_over_ranks((time.perf_counter() - t0) / args.steps, world, dev)
        # the value is the mean over the steps; single calls vary with the host
        # side of the copies (reported beside it)
        e2e = {"value": job_rate(n, world, e2e_s), "unit": UNIT, "h2d_bytes_per_step": int(hq.numel() * 8),
               "d2h_bytes_per_step": int(hi.numel() * 8), "form": head,
               "ms_per_step": {"mean": 1e3 * e2e_s, "median": 1e3 * float(np.median(per)),
                               "min": 1e3 * min(per), "max": 1e3 * max(per)}}
    for r in res.values():
        L.poro_destroy(r["ctx"])
    steps = serving = None
    if not args.no_steps and world == 1:
        try:
            steps = time_stepping_sections(L, local, args)
        except Exception as ex:  # reported, the headline line still prints
            steps = {"error": repr(ex)}
    if not args.no_serving and world == 1:
        try:
            serving = serving_section(L, local, args)
        except Exception as ex:
            serving = {"error": repr(ex)}
    lu = None
    if not args.no_lu and world == 1:
        lu = lu_comparator(L, torch, dev, local, args, float(peaks["hbm_gbs"]))
    sweeps = None
    if not args.no_sweeps and world == 1:
        try:
            sweeps = predictor_sweeps(L, torch, dev, local, args, d)
        except Exception as ex:
            sweeps = {"error": repr(ex)}

    systems = None
    if not args.no_systems and world == 1:
        try:
            systems = other_systems(L, torch, dev, local, args)
        except Exception as ex:
            systems = {"error": repr(ex)}

    if rank != 0:
        if world > 1:
            dist.barrier()
            dist.destroy_process_group()
        return
    cpu = None
    if world == 1 and not args.no_cpu:
        cpu = cpu_baseline(args)
    forms_out = {}
    for name, r in res.items():
        forms_out[name] = {"value": job_rate(n, world, r["ms"] * 1e-3), "ms_per_step": r["ms"],
                           "refine_sweeps": r["sweeps"] if name != "fp64" else None,
                           "roofline": roofline(name), "clocks": r["clocks"]}
        if name in errs:
            forms_out[name]["error_vs_fp64"] = errs[name]
    cfg = _workload(args)
    cfg["form"] = head
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": hr["ms"], "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "data": "synthetic",
        # one refinement sweep: double-binary32 with integer Khat sums
        "dtype": "f64" if head == "fp64" or hr["sweeps"] == 2 else "f32x2+i64" if hr["sweeps"] == 1 else
                 {"mixed": "tf32x3+f32", "mixed_bf16x3": "bf16x3+f32"}[head],
        "config": cfg, "roofline": roofline(head), "forms": forms_out, "mixed_error": errs.get(head),
        "cpu_baseline": cpu, "e2e": e2e, "clocks": hr["clocks"], "gpu_launches": args.steps,
        "lu_comparator": lu, "predictor_sweeps": sweeps, "other_systems": systems, "time_stepping": steps,
        "serving": serving,
    }
    print(json.dumps(out))
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()


def run_planewave_study(args):
    """The paper's plane-wave convergence experiment (Section "Convergence")
    at scale on the GPU: fast P + two S waves of the Biot system (k = (pi, pi,
    pi)) on the periodic cube [-1, 1]^3 cut into 6 n^3 Kuhn tetrahedra, global
    time stepping to t ~ 1e-4 s, L1 / L2 / L-infinity errors against the
    exact solution and their rates between successive meshes, N = 1..6.
    Prints one JSON line (not the benchmark's headline)."""
    import torch

    from oracle import planewave
    from paper_2108_10565_gb300 import _lib as L
    from paper_2108_10565_gb300 import inputs

    torch.cuda.set_device(0)
    K = np.array([np.pi, np.pi, np.pi])
    md = inputs.material_dict(inputs.REFERENCE_MATERIAL)
    modes = planewave.plane_wave_modes(md, K, 3)
    meshes = {1: (4, 8, 16, 32, 64), 2: (4, 8, 16, 32, 64), 3: (4, 8, 16, 32), 4: (4, 8, 16, 32), 5: (4, 8, 16),
              6: (4, 8, 16)}
    out = {"experiment": "plane-wave convergence, periodic cube [-1,1]^3, 6 n^3 tets, t_end ~ 1e-4 s, FP64",
           "degrees": {}}
    for N in sorted(meshes):
        if N not in args.planewave_degrees:
            continue
        rows = []
        for n in meshes[N]:
            mesh = inputs.kuhn_box_mesh(n, lo=(-1, -1, -1), hi=(1, 1, 1))
            ne = len(mesh["tets"])
            v = mesh["vertices"][mesh["tets"]]
            t0 = time.perf_counter()
            ctx = L.poro_create(0, N, L.PORO_FP64)
            try:
                L.poro_set_mesh(ctx, mesh["vertices"], mesh["tets"], mesh["neighbors"], mesh["face_tag"])
                L.poro_set_materials(ctx, np.tile(inputs.REFERENCE_MATERIAL, (ne, 1)))
                dt, _ = L.poro_set_clusters(ctx, 0.5, 1)
                L.poro_set_dofs(ctx, planewave.project(v, N, lambda x: planewave.plane_wave(x, 0.0, K, modes)))
                t1 = time.perf_counter()
                L.poro_advance(ctx, 1e-4)
                t_run = time.perf_counter() - t1
                Q = L.poro_get_dofs(ctx)
                t, _ = L.poro_get_time(ctx)
            finally:
                L.poro_destroy(ctx)
            nr = planewave.error_norms(v, N, Q, lambda x: planewave.plane_wave(x, t, K, modes))
            rel = [a / b for a, b in zip(nr["err"], nr["ref"])]
            rows.append({"n": n, "elements": ne, "steps": int(round(t / dt)), "t": t, "rel_L1": rel[0],
                         "rel_L2": rel[1], "rel_Linf": rel[2], "gpu_advance_s": t_run,
                         "total_s": time.perf_counter() - t0})
        for a, b in zip(rows[:-1], rows[1:]):
            b["rates"] = {k: float(np.log2(a[f"rel_{k}"] / b[f"rel_{k}"])) for k in ("L1", "L2", "Linf")}
        out["degrees"][str(N)] = rows
        print(json.dumps({"N": N, "rows": rows}), file=sys.stderr, flush=True)
    print(json.dumps(out))


def main():
    args = parse()
    if args.planewave_study:
        run_planewave_study(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
