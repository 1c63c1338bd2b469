#!/usr/bin/env python
"""Benchmark of the GB300 messenger-field Wiener filter.

Workload: HEALPix temperature map, nside 2048 (50,331,648 pixels), lmax 4096,
CMB-like C_l with a 5' beam, noise dynamic range 1e4 from the hit pattern,
galactic cut |b| < 15 deg plus 3000 point-source disks of 0.3 deg (synthetic
stand-in for a Planck-resolution map).  One step = one complete Wiener-filter
solve (setup, cooling schedule with band-limited transforms, lambda = 1
iterations down to the residual tolerance, output map) in mixed precision,
with inputs resident in HBM.

Reported (one JSON line on rank 0):
  value       messenger iterations per second over the timed solves (all ranks)
  ms_per_step time to solution of one solve
  roofline    the dominant kernel (Legendre) against the FP32 ALU peak
  e2e         the same metric through wf_solve_host (host buffers, copies timed)
  fp64_path   the plain FP64 GPU path on the same GB300 (full-band iteration
              rate measured; its time to solution extrapolated from it)
  cpu_baseline  the FP64 CPU oracle on a bounded sample of one iteration

--impl reference runs the oracle (the only reference implementation there is)
on the host cores on a bounded sample of the same workload.
"""
import argparse
import json
import math
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import wf_inputs as gen  # noqa: E402

CFG = {"workload": "healpix_T_nside2048_lmax4096", "nside": 2048, "lmax": 4096, "fwhm_arcmin": 5.0,
       "noise_range": 1e4, "b_cut_deg": 15.0, "n_disks": 3000, "disk_radius_deg": 0.3}
METRIC = "messenger iterations/s, full Wiener-filter solve to residual tol (HEALPix nside 2048, lmax 4096)"
UNIT = "iter/s"
FP32_LANES_PER_SM = 128  # FP32 FMA lanes per SM (GB300)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--precision", default="mixed", choices=["mixed", "fp64", "tf32", "bf16"],
                    help="mixed: FP32 Legendre kernels (the workload's default); tf32 / bf16: the same with the "
                         "synthesis on the tensor cores (3xTF32 / split BF16); fp64: the FP64 path")
    ap.add_argument("--tol", type=float, default=None,
                    help="relative residual at which a solve stops (default 1e-6 on the flat grid, 1e-4 on the "
                         "HEALPix workloads, where 1e-6 is out of reach of the messenger iteration: its residual "
                         "tail decays as a power law)")
    ap.add_argument("--maxiter", type=int, default=3000, help="iteration cap of one solve (one step)")
    ap.add_argument("--mixed-correction", type=float, default=1.5,
                    help="mixed precision: at lambda = 1 on the full band, once the residual is below tol x this, "
                         "one FP64 step and then the FP32 iteration on the correction to that step's iterate "
                         "(0: off)")
    ap.add_argument("--mixed-tol-factor", type=float, default=0.98,
                    help="mixed precision: the FP32 iteration stops at tol x factor, then FP64 sweeps check the "
                         "result against tol under the FP64 operator")
    ap.add_argument("--refine-sweeps", type=int, default=6,
                    help="at most this many FP64 lambda = 1 correction sweeps after the mixed iteration; they stop "
                         "once the FP64 operator's residual is below tol (0: none)")
    ap.add_argument("--schedule", default="heuristic", choices=["heuristic", "bound"],
                    help="cooling: the heuristic of Sect. 3 (default) or the chi^2 bound of Sect. 2.2")
    ap.add_argument("--nside", type=int, default=CFG["nside"])
    ap.add_argument("--lmax", type=int, default=CFG["lmax"])
    ap.add_argument("--no-fp64", action="store_true", help="skip the FP64-path comparison")
    ap.add_argument("--no-cpu", action="store_true", help="skip the oracle CPU baseline")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--serve", action="store_true",
                    help="serving workload instead: Poisson stream of mixed-size requests through wf_server_*")
    ap.add_argument("--serve-requests", type=int, default=2000)
    ap.add_argument("--serve-rate", type=float, default=50.0, help="offered requests per second")
    ap.add_argument("--serve-slots", type=int, default=8)
    ap.add_argument("--serve-budget-gb", type=float, default=64.0)
    ap.add_argument("--serve-maxiter", type=int, default=3000)
    ap.add_argument("--no-autotune", action="store_true", help="keep the default Legendre tiles")
    ap.add_argument("--pol-batch", type=int, default=0,
                    help="batched polarised constrained realisations of this many (I, Q, U) maps")
    ap.add_argument("--pol-nsides", default="32,64,128", help="nside choices of the polarised maps (lmax = 2 nside)")
    ap.add_argument("--pol-tol", type=float, default=1e-4)
    ap.add_argument("--pol-maxiter", type=int, default=3000)
    ap.add_argument("--pol-precision", default="mixed", choices=["mixed", "fp64", "tf32", "bf16"],
                    help="tf32 / bf16: the T and spin-2 syntheses on the tensor cores, maps of one nside "
                         "sharing one launch per step")
    ap.add_argument("--pol-no-alone", action="store_true", help="time the batch only (no one-by-one comparison)")
    ap.add_argument("--batch", type=int, default=0,
                    help="batching workload instead: this many solves of mixed nside (64-256), "
                         "run one by one and as one wf_solve_batch")
    ap.add_argument("--config", type=int, default=3, choices=[1, 2, 3],
                    help="1: flat 128x128 FP64 (us per iteration, time to tol); 2: HEALPix nside 512 / lmax 1024 "
                         "FP64 (time to tol, p50/p99); 3: the nside 2048 headline (default)")
    ap.add_argument("--columns", type=int, default=0,
                    help="many maps of one geometry: N maps of one noise model, each a Wiener filter plus a "
                         "fluctuation solve (2N batch columns), tensor-core (tf32) plans against FP32 plans")
    ap.add_argument("--columns-nside", type=int, default=1024)
    ap.add_argument("--columns-iters", type=int, default=30,
                    help="full-band lambda = 1 iterations per timed batch (0: solve every column to --tol)")
    ap.add_argument("--full-band-iters", type=int, default=0,
                    help="replay this many lambda = 1, L = lmax iterations instead of the cooling schedule "
                         "(steady-state timing and profiling)")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def aggregate_over_ranks(t_ms, units, device):
    """Whole-job figures of independent replicas: the slowest rank's time (all
    ranks start after one barrier and stop before another) and the units of
    work all ranks processed.  Works on any initialised process group (NCCL on
    the GPUs, gloo in the CPU tests); one rank returns its own figures."""
    import torch
    import torch.distributed as dist

    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(t_ms), float(units)
    t = torch.tensor([float(t_ms)], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t[0]), float(u[0])


def make_problem(nside, lmax, k):
    kw = dict(fwhm_arcmin=CFG["fwhm_arcmin"], b_cut_deg=CFG["b_cut_deg"], n_disks=CFG["n_disks"],
              disk_radius_deg=CFG["disk_radius_deg"], noise_range=CFG["noise_range"])
    return gen.healpix_problem(nside, lmax, gen.seed_for(3, k), **kw)


# --------------------------------------------------------------------------
# algorithmic work of the Legendre transforms (per full launch)
# --------------------------------------------------------------------------
def legendre_triples(nside, L):
    """(l, m, ring-pair) triples of one Legendre transform at band limit L."""
    npairs = 2 * nside
    return npairs * (L + 1) * (L + 2) // 2


LEG_FLOPS_PER_TRIPLE = 7  # recurrence (mul + fma = 3 flops) + contraction (2 fma = 4 flops)


def peak_fp32_tflops(mhz, n_sm):
    """FP32 FMA peak from unit counts: SMs x 128 lanes x 2 flops x clock."""
    return n_sm * FP32_LANES_PER_SM * 2 * mhz * 1e6 / 1e12


def time_to_residual(rep):
    """Device time (s) from the start of the solve until the relative residual
    first falls below each tolerance (None if it does not within the solve)."""
    ms = np.nan_to_num(rep["iter_ms_trace"], nan=0.0)
    cum = np.cumsum(ms) / 1e3
    res = rep["resid_trace"]
    out = {}
    for tol in (1e-2, 1e-3, 1e-4, 1e-5, 1e-6):
        hit = np.nonzero(res < tol)[0]
        out["%g" % tol] = {"s": float(cum[hit[0]]), "iters": int(hit[0] + 1)} if hit.size else None
    return out


def time_to_dchi2(rep, lmax):
    """The paper's own stopping rule (Sect. 3): the first lambda = 1, full-band
    iteration whose chi^2 changed by less than 1e-4 sigma_chi2 = 1e-4 sqrt(2
    n_dof); device time, iteration and the relative residual there."""
    ms = np.nan_to_num(rep["iter_ms_trace"], nan=0.0)
    cum = np.cumsum(ms) / 1e3
    chi, lam, L, res = rep["chi2_trace"], rep["lambda_trace"], rep["L_trace"], rep["resid_trace"]
    sig = math.sqrt(2.0 * rep["n_dof"])
    full = (lam == 1.0) & (L == lmax)
    for k in range(1, len(chi)):
        if full[k] and full[k - 1] and abs(chi[k] - chi[k - 1]) < 1e-4 * sig:
            return {"s": float(cum[k]), "iters": int(k + 1), "residual": float(res[k])}
    return None


# --------------------------------------------------------------------------
# clocks sampling during the timed region
# --------------------------------------------------------------------------
class Clocks:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = gpu_index
        self.f = tempfile.NamedTemporaryFile(mode="w+", suffix=".csv", delete=False)
        self.p = None

    def start(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), "--query-gpu=" + self.Q,
                                       "--format=csv,noheader,nounits", "-lms", "200"], stdout=self.f,
                                      stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.p.kill()
        self.f.flush()
        self.f.seek(0)
        sm, smax, reasons, power = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.f.read().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
                power.append(float(parts[3]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        os.unlink(self.f.name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(smax)), "reasons": sorted(reasons),
                "power_w_max": float(max(power)), "samples": len(sm)}


# --------------------------------------------------------------------------
# CPU oracle on a bounded sample of one full-band iteration
# --------------------------------------------------------------------------
def oracle_iteration_sample(nside, lmax, n_rings=8, n_m=8, seed=0, keep=False):
    """Time the oracle's synthesis on n_rings evenly spaced rings and its
    adjoint on n_m evenly spaced m, both at the full band, and extrapolate to
    one messenger iteration (one synthesis of every ring + one adjoint of
    every m; the blends are negligible).  Returns (seconds/iteration, sample
    description, threads, sample): with ``keep`` the sample holds the inputs
    and the oracle's outputs, so that the GPU's transforms of the same inputs
    can be compared with them."""
    import oracle

    rng = np.random.default_rng(seed)
    a = gen.alm_unit_gaussian(rng, lmax) * np.sqrt(gen.cmb_like_cl(lmax, 5.0)[gen.alm_ell(lmax)] + 1e-30)
    R = 4 * nside - 1
    rings = np.linspace(0, R - 1, n_rings).round().astype(int)
    syn = []
    t0 = time.perf_counter()
    for r in rings:
        syn.append(oracle.synthesis(nside, lmax, lmax, a, rings=(int(r), int(r) + 1)))
    t_ring = (time.perf_counter() - t0) / n_rings
    f = rng.standard_normal(12 * nside * nside)
    ms = np.linspace(0, lmax, n_m).round().astype(int)
    adj = []
    t0 = time.perf_counter()
    for m in ms:
        adj.append(oracle.adjoint_synthesis(nside, lmax, lmax, f, ms=(int(m), int(m) + 1)))
    t_m = (time.perf_counter() - t0) / n_m
    t_iter = t_ring * R + t_m * (lmax + 1)
    desc = ("oracle synthesis of %d evenly spaced rings and adjoint of %d evenly spaced m at nside %d, lmax %d, "
            "extrapolated to one full-band iteration (%d rings, %d m)" % (n_rings, n_m, nside, lmax, R, lmax + 1))
    sample = {"a": a, "rings": rings, "syn": syn, "f": f, "ms": ms, "adj": adj} if keep else None
    return t_iter, desc, oracle.num_threads(), sample


def ring_slices(nside, rings):
    """Pixel ranges of the given RING-order rings."""
    _, _, nr = gen.ring_layout(nside)
    off = np.concatenate([[0], np.cumsum(nr)])
    return [slice(int(off[r]), int(off[r + 1])) for r in rings]


def sampled_errors(sample, nside, lmax, gpu_map, gpu_alm):
    """Max relative error of the GPU's synthesis on the sampled rings and of its
    adjoint on the sampled m, against the oracle's values there."""
    sl = ring_slices(nside, sample["rings"])
    num = max(float(np.max(np.abs(gpu_map[s] - o[s]))) for s, o in zip(sl, sample["syn"]))
    den = max(float(np.max(np.abs(o[s]))) for s, o in zip(sl, sample["syn"]))
    e_syn = num / den
    num = den = 0.0
    for m, o in zip(sample["ms"], sample["adj"]):
        i0 = int(m) * (2 * lmax + 3 - int(m)) // 2
        i1 = i0 + lmax + 1 - int(m)
        num = max(num, float(np.max(np.abs(gpu_alm[i0:i1] - o[i0:i1]))))
        den = max(den, float(np.max(np.abs(o[i0:i1]))))
    return e_syn, num / den


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    import oracle  # noqa: F401  (builds the C core if needed)

    for _ in range(args.warmup):
        oracle_iteration_sample(args.nside, args.lmax, n_rings=2, n_m=2)
    ts, walls = [], []
    desc, thr = "", 1
    for k in range(args.steps):
        w0 = time.perf_counter()
        t, desc, thr, _ = oracle_iteration_sample(args.nside, args.lmax, n_rings=4, n_m=4, seed=k)
        walls.append(time.perf_counter() - w0)
        ts.append(t)
    t = float(np.mean(ts))
    v = 1.0 / t
    # each step times a bounded sample (a few rings and m) and extrapolates it to one iteration: the
    # rate is an extrapolated per-iteration rate, and no full step of the workload is run
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": None,
            "ms_per_iteration_extrapolated": t * 1e3, "sample_s_per_step": float(np.mean(walls)),
            "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": CFG["workload"], "nside": args.nside, "lmax": args.lmax,
                       "implementation": "FP64 CPU oracle (direct Legendre and Fourier sums), per-iteration rate"},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": thr, "kind": "oracle", "sample": desc},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# --------------------------------------------------------------------------
# GPU arm
# --------------------------------------------------------------------------
def run_ours(args):
    import torch

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=dev)
    import paper_1210_4931_gb300 as wf

    wf.load()
    nside, lmax = args.nside, args.lmax
    P = make_problem(nside, lmax, rank)
    stream = torch.cuda.current_stream()
    plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=args.precision)
    tiles = wf.wf_plan_tiles(plan) if args.no_autotune else wf.wf_plan_autotune(plan)
    T = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    # data = signal (synthesised by the library's own basis change) + noise
    a_sig = T(P["a_signal"])
    s_sig = torch.empty(plan.npix, dtype=torch.float64, device=dev)
    wf.wf_alm2map(plan, a_sig, lmax, s_sig)
    d = s_sig + T(P["noise"])
    nv, mask, cl = T(P["noise_var"]), T(P["mask"]), T(P["c_ell"])
    s_out = torch.empty(plan.npix, dtype=torch.float64, device=dev)
    alm_out = torch.empty(plan.nalm, dtype=torch.complex128, device=dev)
    sched = 1 if args.schedule == "bound" else 0
    wf.wf_set_options(plan, profile=1, maxiter=args.maxiter, schedule=sched,
                      refine_sweeps=args.refine_sweeps if args.precision != "fp64" else 0,
                      mixed_tol_factor=args.mixed_tol_factor,
                      mixed_correction=args.mixed_correction if args.precision != "fp64" else 0.0)
    if args.full_band_iters > 0:
        wf.wf_set_schedule(plan, [1.0] * args.full_band_iters, [lmax] * args.full_band_iters)
    cap = max(args.maxiter, args.full_band_iters) + 16

    def solve():
        return wf.wf_solve(plan, d, nv, mask, cl, args.tol, s_out, alm_out, trace_cap=cap)

    for _ in range(args.warmup):
        solve()
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    clocks = Clocks(local)
    clocks.start()
    reps = []
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(args.steps):
        reps.append(solve())
    e1.record(stream)
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    ck = clocks.stop()
    t_ms = e0.elapsed_time(e1)
    iters = sum(r["iters"] for r in reps)
    t_ms, iters = aggregate_over_ranks(t_ms, iters, dev)
    value = iters / (t_ms / 1e3)
    last = reps[-1]

    # per-iteration times (p50/p99) at the full band, lambda = 1
    full = (last["lambda_trace"] == 1.0) & (last["L_trace"] == lmax)
    nsw = [int(r.get("refine_sweeps") or 0) for r in reps]

    def switch_index(r):
        # the correction form's FP64 step: the first iteration with no chi^2 (-1: no switch)
        nan = np.flatnonzero(np.isnan(r["chi2_trace"]))
        return int(nan[0]) if nan.size and args.precision != "fp64" and args.mixed_correction > 0 else -1

    def fp32_full_band(r, k):
        # the mixed path's own full-band lambda = 1 iterations: no FP64 sweep, no FP64 switch step
        n = len(r["iter_ms_trace"]) - k
        sel = (r["lambda_trace"][:n] == 1.0) & (r["L_trace"][:n] == lmax)
        j = switch_index(r)
        if 0 <= j < n:
            sel[j] = False
        return r["iter_ms_trace"][:n][sel]

    it_ms = np.concatenate([fp32_full_band(r, k) for r, k in zip(reps, nsw)])
    all_ms = np.concatenate([r["iter_ms_trace"] for r in reps])
    sw = switch_index(last)

    # roofline of the dominant kernel: Legendre synthesis + analysis (FP32 ALU)
    kms = {k: sum(r["kernel_ms"][k] for r in reps) for k in reps[0]["kernel_ms"]}
    kl = {k: sum(r["kernel_launches"][k] for r in reps) for k in reps[0]["kernel_launches"]}
    leg_triples = 0
    for r in reps:
        for L in r["L_trace"]:
            leg_triples += 2 * legendre_triples(nside, int(L))  # synthesis + analysis
    leg_ms = kms["leg_syn"] + kms["leg_ana"]
    achieved = LEG_FLOPS_PER_TRIPLE * leg_triples / (leg_ms / 1e3) / 1e12
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    peak_units = peak_fp32_tflops(2070.0, n_sm)
    # the measured FP32 FMA rate of this GPU (packed f32x2 FMAs, as the kernels issue them)
    peak_meas = {"packed": wf.wf_probe_fp32_fma(True), "scalar": wf.wf_probe_fp32_fma(False)}
    peak = max(peak_meas.values())
    # DRAM bytes (read + write) of one full-band k_legsyn_mx<8> + k_legana_mx<8> + k_ana_epilogue at
    # nside 2048, lmax 4096, from a one-pass ncu capture of these kernels (924.8 + 641.7 + 702.2 MB);
    # other sizes or tiles were not captured
    traffic = 2268670000 if (nside, lmax, tuple(tiles), args.precision) == (2048, 4096, (8, 8), "mixed") else None
    roof = {"bound": "alu", "kernel": "legendre synthesis + analysis (k_legsyn, k_legana)",
            "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak, "traffic": traffic,
            "traffic_basis": "DRAM bytes of one full-band synthesis + analysis pair (ncu dram__bytes_read.sum + "
                             "dram__bytes_write.sum)" if traffic else None,
            "peak_basis": "measured: FP32 FMA loop (wf_probe_fp32_fma, best of packed f32x2 and scalar FMAs) "
                          "in this process, %.1f / %.1f TFLOP/s; from unit counts %d SMs x 128 lanes x 2 flop x "
                          "2070 MHz = %.1f TFLOP/s" % (peak_meas["packed"], peak_meas["scalar"], n_sm, peak_units),
            "peak_units_tflops": peak_units,
            "flops_per_triple": LEG_FLOPS_PER_TRIPLE, "kernel_ms": leg_ms,
            "note": "the synthesis runs on the tensor cores: the FP32 peak bounds the analysis only"
                    if args.precision in ("tf32", "bf16") else None,
            "share_of_step": leg_ms / max(1e-9, sum(kms.values()))}

    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": t_ms / args.steps, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": {"mixed": "f32+f64", "fp64": "f64", "tf32": "tf32x3+f32+f64",
                                            "bf16": "bf16x3+f32+f64"}[args.precision], "data": "synthetic",
           "config": {"workload": CFG["workload"], "nside": nside, "lmax": lmax, "precision": args.precision,
                      "tol": args.tol, "schedule": args.schedule, "legendre_tiles": list(tiles),
                      "tol_check": "the result's residual under the FP64 operator (correction sweeps); the FP32 "
                                   "iteration (in correction form once lambda = 1 and its residual is below %g x "
                                   "tol) stops at %g x tol, then at most %d sweeps"
                                   % (args.mixed_correction, args.mixed_tol_factor, args.refine_sweeps)
                                   if args.precision != "fp64" and args.refine_sweeps > 0 else "own operator",
                      "l2": "inputs (1.2 GB) larger than L2",
                      "parallelism": "replicas"},
           "time_to_tol_s": t_ms / args.steps / 1e3 if last["converged"] else None,
           "time_to_residual_s": time_to_residual(last),
           "time_to_paper_stop_s": time_to_dchi2(last, lmax),
           "iters_per_solve": last["iters"],
           "maxiter": args.maxiter, "mixed_lc": last.get("mixed_lc"), "fp64_sweeps": last.get("refine_sweeps"),
           "correction_switch": {"iter": sw, "fp64_step_ms": float(last["iter_ms_trace"][sw]),
                                 "fp64_residual_at_switch": float(last["resid_trace"][sw])} if sw >= 0 else None,
           "final_residual": last["final_residual"], "converged": last["converged"],
           "chi2_over_ndof": last["chi2_over_ndof"],
           "iter_ms_full_band": {"p50": float(np.percentile(it_ms, 50)) if it_ms.size else None,
                                 "p99": float(np.percentile(it_ms, 99)) if it_ms.size else None,
                                 "n": int(it_ms.size)},
           "iter_ms_all": {"p50": float(np.percentile(all_ms, 50)), "p99": float(np.percentile(all_ms, 99))},
           "kernel_ms_per_step": {k: v / args.steps for k, v in kms.items()},
           "gpu_launches": int(sum(r["launches"] for r in reps)),
           "roofline": roof, "clocks": ck}

    if rank == 0 and not args.no_e2e:
        # e2e: host buffers in, host map out, through wf_solve_host; the buffers are pinned
        # (page-locked) host memory, so the copies run as DMA at the link's rate
        def pinned(a):
            t = torch.empty(a.shape, dtype=getattr(torch, str(a.dtype)), pin_memory=True)
            t.numpy()[...] = a
            return t.numpy()

        dh = pinned(d.cpu().numpy())
        nvh, mh, clh = pinned(P["noise_var"]), pinned(P["mask"]), pinned(P["c_ell"])
        sh = torch.empty(plan.npix, dtype=torch.float64, pin_memory=True).numpy()
        wf.wf_set_options(plan, profile=0, maxiter=args.maxiter, schedule=sched,
                          refine_sweeps=args.refine_sweeps if args.precision != "fp64" else 0,
                          mixed_tol_factor=args.mixed_tol_factor,
                          mixed_correction=args.mixed_correction if args.precision != "fp64" else 0.0)
        wf.wf_solve_host(plan, dh, nvh, mh, clh, args.tol, sh)  # warm
        t0 = time.perf_counter()
        rep = wf.wf_solve_host(plan, dh, nvh, mh, clh, args.tol, sh)
        te = time.perf_counter() - t0
        out["e2e"] = {"value": rep["iters"] / te, "unit": UNIT,
                      "h2d_bytes_per_step": int(dh.nbytes + nvh.nbytes + mh.nbytes + clh.nbytes),
                      "d2h_bytes_per_step": int(sh.nbytes), "seconds_per_solve": te,
                      "host_buffers": "pinned"}
    if rank == 0 and ws == 1 and not args.no_cpu:
        # the oracle on a bounded sample of one iteration (timed), and the GPU's transforms of the
        # same inputs compared with the oracle's values on the sampled rings and m
        import oracle

        t_it, desc, thr, smp = oracle_iteration_sample(nside, lmax, n_rings=8, n_m=8, keep=True)
        out["cpu_baseline"] = {"value": 1.0 / t_it, "unit": UNIT, "cores": thr, "kind": "oracle", "sample": desc}
        gm = torch.empty(plan.npix, dtype=torch.float64, device=dev)
        wf.wf_alm2map(plan, T(smp["a"]), lmax, gm)
        ga = torch.empty(plan.nalm, dtype=torch.complex128, device=dev)
        wf.wf_map2alm_adjoint(plan, T(smp["f"]), lmax, ga)
        e_syn, e_adj = sampled_errors(smp, nside, lmax, gm.cpu().numpy(), ga.cpu().numpy())
        # the returned map against the oracle's synthesis of the returned a_lm (polar, cap edge,
        # equator and southern belt rings)
        a_fin, s_fin = alm_out.cpu().numpy(), s_out.cpu().numpy()
        rr = [0, nside - 1, 2 * nside - 1, 3 * nside]
        ref = [oracle.synthesis(nside, lmax, lmax, a_fin, rings=(r, r + 1)) for r in rr]
        sl = ring_slices(nside, rr)
        e_map = (max(float(np.max(np.abs(s_fin[q] - o[q]))) for q, o in zip(sl, ref)) /
                 max(float(np.max(np.abs(o[q]))) for q, o in zip(sl, ref)))
        out["err_vs_oracle"] = {
            "synthesis_sampled_rings": e_syn, "adjoint_sampled_m": e_adj,
            "result_map_vs_oracle_synthesis_of_result_alm": e_map,
            "result_relative_residual": last["final_residual"],
            "basis": "max |GPU - oracle| / max |oracle|: the plan's (%s) synthesis of a CMB-like a_lm on rings %s, "
                     "its adjoint of a white map on m %s, and the returned s_WF on rings %s against the oracle's "
                     "synthesis of the returned a_lm; the residual is the solve's own relative residual"
                     % (args.precision, [int(r) for r in smp["rings"]], [int(m) for m in smp["ms"]], rr)}
    plan.close()
    del plan

    if rank == 0 and not args.no_fp64 and args.precision == "mixed":
        p64 = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="fp64")
        wf.wf_set_options(p64, profile=1)
        nrep = 3
        wf.wf_set_schedule(p64, [1.0] * nrep, [lmax] * nrep)
        wf.wf_solve(p64, d, nv, mask, cl, args.tol, s_out, trace_cap=16)  # warm
        r64 = wf.wf_solve(p64, d, nv, mask, cl, args.tol, s_out, trace_cap=16)
        ms64 = float(np.mean(r64["iter_ms_trace"][:nrep]))
        # extrapolate the FP64 time to solution along the mixed solve's own trace
        Ls = last["L_trace"]
        cost = float(np.sum((Ls.astype(np.float64) + 1) ** 2) / (lmax + 1) ** 2)
        out["fp64_path"] = {"iters_per_s_full_band": 1e3 / ms64, "iter_ms_full_band": ms64,
                            # the FP64 path needs the same iterations (its residual trace follows the mixed
                            # one); a time to tol only exists where the mixed solve reached tol
                            "time_to_tol_s_extrapolated": ms64 * cost / 1e3 if last["converged"] else None,
                            "time_same_trace_s_extrapolated": ms64 * cost / 1e3,
                            "speedup_mixed_vs_fp64_full_band":
                                ms64 / out["iter_ms_full_band"]["p50"] if out["iter_ms_full_band"]["p50"] else None,
                            "note": "FP64 full-band iteration measured (3 iterations, lambda = 1); its time "
                                    "over the mixed solve's own (lambda, L) trace extrapolated with cost "
                                    "proportional to (L+1)^2"}
        p64.close()

    if rank == 0:
        print(json.dumps(out))
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


# --------------------------------------------------------------------------
# serving workload: Poisson stream of Wiener-filter requests of mixed size
# --------------------------------------------------------------------------
SERVE_NSIDES = [64, 128, 256, 512, 1024]
SERVE_WEIGHTS = [0.3, 0.3, 0.2, 0.15, 0.05]
SERVE_POOL = {64: 6, 128: 6, 256: 4, 512: 3, 1024: 2}  # distinct seeded problems per nside


def serve_problems(wf, dev):
    """Seeded problems per nside: power-law C_l = l^-n (n ~ U(2, 3)), hit
    pattern with its own jitter, |b| < U(10, 25) deg plus U{0..1000} disks of
    0.3 deg; data = signal synthesised by the library + noise."""
    import torch

    pool = {}
    for ns in SERVE_NSIDES:
        lmax = 2 * ns
        plan = wf.wf_plan_create("healpix", nside=ns, lmax=lmax, precision="fp64")
        items = []
        for k in range(SERVE_POOL[ns]):
            rng = np.random.default_rng(gen.seed_for(5, 100 * ns + k))
            cl = gen.power_law_cl(lmax, float(rng.uniform(2.0, 3.0)))
            P = gen.healpix_problem(ns, lmax, gen.seed_for(5, 100 * ns + 50 + k), cl=cl,
                                    b_cut_deg=float(rng.uniform(10.0, 25.0)), n_disks=int(rng.integers(0, 1001)),
                                    disk_radius_deg=0.3)
            s = torch.empty(plan.npix, dtype=torch.float64, device=dev)
            wf.wf_alm2map(plan, torch.from_numpy(P["a_signal"]).to(dev), lmax, s)
            d = s.cpu().numpy() + P["noise"]
            items.append({"d": np.ascontiguousarray(d), "noise_var": np.ascontiguousarray(P["noise_var"]),
                          "mask": np.ascontiguousarray(P["mask"]), "C_ell": np.ascontiguousarray(cl)})
        plan.close()
        pool[ns] = items
    return pool


def run_serve(args):
    import torch

    import paper_1210_4931_gb300 as wf

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    wf.load()
    pool = serve_problems(wf, dev)
    rng = np.random.default_rng(gen.seed_for(5, 7))
    n = args.serve_requests
    gaps = rng.exponential(1.0 / args.serve_rate, n)
    arrive = np.cumsum(gaps) - gaps[0]
    ns_of = rng.choice(SERVE_NSIDES, size=n, p=SERVE_WEIGHTS)
    prob_of = [int(rng.integers(0, SERVE_POOL[int(x)])) for x in ns_of]
    tol_of = rng.choice([1e-4, 1e-6], size=n)
    free = {ns: [] for ns in SERVE_NSIDES}  # recycled output maps
    srv = wf.Server(device=local, mem_budget=int(args.serve_budget_gb * (1 << 30)), slots=args.serve_slots)
    outs, results = {}, {}
    clocks = Clocks(local)
    clocks.start()
    t0 = time.perf_counter()
    i = 0
    while len(results) < n:
        now = time.perf_counter() - t0
        while i < n and arrive[i] <= now:
            ns = int(ns_of[i])
            R = pool[ns][prob_of[i]]
            out = free[ns].pop() if free[ns] else np.empty(12 * ns * ns)
            outs[i] = (ns, out)
            srv.submit("wf", nside=ns, lmax=2 * ns, precision="mixed", tol=float(tol_of[i]), s_out=out, tag=i,
                       d=R["d"], noise_var=R["noise_var"], mask=R["mask"], C_ell=R["C_ell"],
                       maxiter=args.serve_maxiter)
            i += 1
        wait = (arrive[i] - (time.perf_counter() - t0)) if i < n else 0.5
        for r in srv.wait(timeout=max(0.0, min(wait, 0.5))):
            results[r["tag"]] = r
            ns, out = outs.pop(r["tag"])
            free[ns].append(out)
    wall = time.perf_counter() - t0
    ck = clocks.stop()
    st = srv.stats()
    srv.close()
    lat = np.array([r["t_done"] - r["t_submit"] for r in results.values()])
    qwait = np.array([r["t_start"] - r["t_submit"] for r in results.values()])
    t_first = min(r["t_submit"] for r in results.values())
    t_last = max(r["t_done"] for r in results.values())
    per = {}
    for ns in SERVE_NSIDES:
        sel = [r for r in results.values() if int(ns_of[r["tag"]]) == ns]
        if sel:
            l_ns = np.array([r["t_done"] - r["t_submit"] for r in sel])
            per[str(ns)] = {"n": len(sel), "p50_ms": float(np.percentile(l_ns, 50) * 1e3),
                            "p99_ms": float(np.percentile(l_ns, 99) * 1e3),
                            "iters_mean": float(np.mean([r["iters"] for r in sel])),
                            "converged": float(np.mean([r["converged"] for r in sel]))}
    ok = sum(1 for r in results.values() if r["status"] in (wf.WF_OK, wf.WF_ENOCONV))

    def lat_of(sel):
        if not sel:
            return None
        x = np.array([r["t_done"] - r["t_submit"] for r in sel])
        s = np.array([r["t_done"] - r["t_start"] for r in sel])
        return {"n": len(sel), "p50_ms": float(np.percentile(x, 50) * 1e3), "p99_ms": float(np.percentile(x, 99) * 1e3),
                "service_p50_ms": float(np.percentile(s, 50) * 1e3),
                "service_p99_ms": float(np.percentile(s, 99) * 1e3),
                "iters_mean": float(np.mean([r["iters"] for r in sel]))}

    conv = [r for r in results.values() if r["converged"]]
    unconv = [r for r in results.values() if not r["converged"]]
    by_tol = {}
    for t in (1e-4, 1e-6):
        sel = [r for r in results.values() if tol_of[r["tag"]] == t]
        by_tol["%g" % t] = {"n": len(sel), "converged_fraction": float(np.mean([r["converged"] for r in sel]))
                            if sel else None}
    out = {"metric": "serving: Wiener-filter solves per second, Poisson arrivals, mixed nside 64-1024",
           "value": n / (t_last - t_first), "unit": "solves/s", "n_gpus": 1, "higher_is_better": True,
           "latency_ms": {"p50": float(np.percentile(lat, 50) * 1e3), "p99": float(np.percentile(lat, 99) * 1e3),
                          "mean": float(lat.mean() * 1e3)},
           "queue_wait_ms": {"p50": float(np.percentile(qwait, 50) * 1e3),
                             "p99": float(np.percentile(qwait, 99) * 1e3)},
           "offered_rate": args.serve_rate, "achieved_rate": n / (t_last - t_first), "requests": n,
           "ok": ok, "converged_fraction": float(np.mean([r["converged"] for r in results.values()])),
           "latency_converged": lat_of(conv), "latency_not_converged": lat_of(unconv), "by_tol": by_tol,
           "per_nside": per, "wall_s": wall, "dtype": "f32+f64", "data": "synthetic",
           "config": {"workload": "serving_T_nside64-1024_poisson", "slots": args.serve_slots,
                      "budget_gb": args.serve_budget_gb, "maxiter": args.serve_maxiter,
                      "tol": "1e-4 or 1e-6 (equiprobable)", "precision": "mixed",
                      "inputs": "seeded pool of %s problems per nside" % SERVE_POOL},
           "server": st, "clocks": ck}
    if rank == 0:
        print(json.dumps(out))
    return 0


# --------------------------------------------------------------------------
# batching workload: many small solves, one by one vs one wf_solve_batch call
# --------------------------------------------------------------------------
def run_batch(args):
    import torch

    import paper_1210_4931_gb300 as wf

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    wf.load()
    rng = np.random.default_rng(gen.seed_for(4, 0))
    n = args.batch
    nsides = rng.choice([64, 128, 256], size=n)
    T = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    items, geo = [], []
    for i, ns in enumerate(nsides):
        ns = int(ns)
        lmax = 2 * ns
        P = gen.healpix_problem(ns, lmax, gen.seed_for(4, 10 + i), cl=gen.cmb_like_cl(lmax, 5.0 * 2048 / ns),
                                b_cut_deg=20.0, n_disks=100, disk_radius_deg=1.0)
        helper = wf.wf_plan_create("healpix", nside=ns, lmax=lmax, precision="fp64")
        s = torch.empty(helper.npix, dtype=torch.float64, device=dev)
        wf.wf_alm2map(helper, T(P["a_signal"]), lmax, s)
        helper.close()
        items.append({"kind": "wf", "d": s + T(P["noise"]), "noise_var": T(P["noise_var"]), "mask": T(P["mask"]),
                      "C_ell": T(P["c_ell"]), "tol": 1e-5, "s_out": torch.empty_like(s)})
        geo.append((ns, lmax))
    plans = [wf.wf_plan_create("healpix", nside=ns, lmax=l, precision="mixed") for ns, l in geo]
    for pl in plans:
        wf.wf_plan_autotune(pl, reps=2)
    stream = torch.cuda.current_stream()

    def one_by_one():
        reps = []
        for pl, it in zip(plans, items):
            reps.append(wf.wf_solve(pl, it["d"], it["noise_var"], it["mask"], it["C_ell"], it["tol"], it["s_out"]))
        return reps

    def batched():
        return wf.wf_solve_batch(plans, items)

    out = {}
    for name, fn in (("one_by_one", one_by_one), ("batched", batched)):
        fn()  # warm: graphs, pooled tables
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ts = []
        for _ in range(max(1, args.steps)):
            e0.record(stream)
            reps = fn()
            e1.record(stream)
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        iters = sum(r["iters"] for r in reps)
        out[name] = {"ms": float(np.median(ts)), "iters": iters, "solves_per_s": n / (np.median(ts) / 1e3),
                     "iters_per_s": iters / (np.median(ts) / 1e3),
                     "converged": int(sum(r["converged"] for r in reps))}
    res = {"metric": "batched solves: Wiener filters of mixed nside 64-256 per second", "unit": "solves/s",
           "value": out["batched"]["solves_per_s"], "n_gpus": 1, "higher_is_better": True, "batch": n,
           "nsides": [int(x) for x in nsides], "one_by_one": out["one_by_one"], "batched": out["batched"],
           "speedup": out["one_by_one"]["ms"] / out["batched"]["ms"], "dtype": "f32+f64", "data": "synthetic",
           "config": {"workload": "batch_T_nside64-256", "precision": "mixed", "tol": 1e-5,
                      "timing": "CUDA events around the whole call, median of --steps runs"}}
    for pl in plans:
        pl.close()
    if rank == 0:
        print(json.dumps(res))
    return 0


def run_columns(args):
    """N maps of one geometry and noise model (the temperature analogue of the batched
    constrained realisations: each map a Wiener filter plus its fluctuation solve, Sect. 2.3)
    as 2N columns of one wf_solve_batch.  Tensor-core plans (tf32) share one synthesis launch
    per step over up to 16 columns; FP32 plans run their own kernels per column.  A step is
    one batch of --columns-iters full-band lambda = 1 iterations of every column (or, with
    --columns-iters 0, a solve of every column to --tol)."""
    import torch

    import paper_1210_4931_gb300 as wf

    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    wf.load()
    nside = args.columns_nside
    lmax = 2 * nside
    nm = args.columns
    P = gen.healpix_problem(nside, lmax, gen.seed_for(4, 1), fwhm_arcmin=13.0, b_cut_deg=20.0, n_disks=500,
                            disk_radius_deg=0.6)
    T = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    helper = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision="fp64")
    npix = helper.npix
    items = []
    common = {"noise_var": T(P["noise_var"]), "mask": T(P["mask"]), "C_ell": T(P["c_ell"]), "tol": args.tol}
    for j in range(nm):
        rng = np.random.default_rng(gen.seed_for(4, 100 + j))
        a = gen.alm_unit_gaussian(rng, lmax) * np.sqrt(P["c_ell"][gen.alm_ell(lmax)])
        s = torch.empty(npix, dtype=torch.float64, device=dev)
        wf.wf_alm2map(helper, T(a), lmax, s)
        d = s + T(np.sqrt(P["noise_var"]) * rng.standard_normal(npix))
        items.append(dict(common, kind="wf", d=d, s_out=torch.empty(npix, dtype=torch.float64, device=dev)))
        items.append(dict(common, kind="fluct", g1=T(rng.standard_normal(npix)),
                          g2=T(np.ascontiguousarray(gen.alm_unit_gaussian(rng, lmax), dtype=np.complex128)),
                          s_out=torch.empty(npix, dtype=torch.float64, device=dev)))
    helper.close()
    stream = torch.cuda.current_stream()
    out, maps = {}, {}
    clocks = Clocks(0)
    for prec in ("mixed", "tf32"):
        plans = [wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=prec) for _ in items]
        wf.wf_plan_autotune(plans[0], reps=2)
        t0, t1 = wf.wf_plan_tiles(plans[0])
        for pl in plans:
            if args.columns_iters > 0:
                wf.wf_set_schedule(pl, [1.0] * args.columns_iters, [lmax] * args.columns_iters)
            else:
                wf.wf_set_options(pl, maxiter=args.maxiter)
        for _ in range(max(1, args.warmup)):
            wf.wf_solve_batch(plans, items)
        torch.cuda.synchronize()
        if prec == "tf32":
            clocks.start()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ts, reps = [], None
        for _ in range(max(1, args.steps)):
            e0.record(stream)
            reps = wf.wf_solve_batch(plans, items)
            e1.record(stream)
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        if prec == "tf32":
            out["clocks"] = clocks.stop()
        iters = sum(r["iters"] for r in reps)
        t = float(np.median(ts))
        out[prec] = {"ms_per_batch": t, "column_iters": iters, "column_iters_per_s": iters / (t / 1e3),
                     "ms_per_column_iteration": t / iters, "launches_per_batch": int(sum(r["launches"] for r in reps)),
                     "converged": int(sum(r["converged"] for r in reps)), "tiles": [t0, t1]}
        maps[prec] = [it["s_out"].cpu().numpy() for it in items]
        for pl in plans:
            pl.close()
    diff = max(float(np.max(np.abs(a - b)) / np.max(np.abs(b))) for a, b in zip(maps["tf32"], maps["mixed"]))
    res = {"metric": "column iterations/s: %d maps x (Wiener filter + fluctuation) of one geometry, nside %d / "
                     "lmax %d" % (nm, nside, lmax), "unit": "column-iter/s", "value": out["tf32"]["column_iters_per_s"],
           "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "dtype": "f32+f64",
           "data": "synthetic", "columns": 2 * nm,
           "config": {"workload": "columns_T_nside%d_%dmaps" % (nside, nm), "iters_per_batch": args.columns_iters,
                      "tol": args.tol, "recipe": "13' beam, |b| < 20 deg + 500 disks of 0.6 deg, one noise model",
                      "l2": "inputs (%d MB) larger than L2" % (2 * nm * npix * 8 // (1 << 20))},
           "tf32_tensor_core": out["tf32"], "fp32_fma": out["mixed"],
           "speedup_tf32_vs_fp32": out["mixed"]["ms_per_batch"] / out["tf32"]["ms_per_batch"],
           "max_rel_diff_tf32_vs_fp32_maps": diff, "clocks": out.get("clocks")}
    print(json.dumps(res))
    return 0


def run_pol_batch(args):
    """Batched polarised constrained realisations: each (I, Q, U) map is a
    Wiener-filter solve plus a fluctuation solve (s_CR = s_WF + f), the pairs of
    all maps advanced together by wf_solve_batch; against the same solves one
    by one.  Also the per-iteration kernel-family times of one full-band
    polarised iteration at the largest nside."""
    import torch

    import paper_1210_4931_gb300 as wf

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    wf.load()
    rng = np.random.default_rng(gen.seed_for(4, 1))
    n = args.pol_batch
    choices = [int(x) for x in args.pol_nsides.split(",")]
    nsides = rng.choice(choices, size=n)
    T = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    items, geo, base = [], [], {}
    for i, ns in enumerate(nsides):
        ns = int(ns)
        lmax = 2 * ns
        # one noise model and mask per nside, own signal, noise and fluctuation draws per map
        if ns not in base:
            base[ns] = gen.healpix_pol_problem(ns, lmax, gen.seed_for(4, 100 + ns), fwhm_arcmin=5.0 * 2048 / ns,
                                               corr=0.1, b_cut_deg=20.0, n_disks=100, disk_radius_deg=1.0,
                                               draws=False)
        P = dict(base[ns], **gen.healpix_pol_draws(base[ns], gen.seed_for(4, 1000 + i)))
        helper = wf.wf_plan_create("healpix", nside=ns, lmax=lmax, precision="fp64", ncomp=3)
        sig = torch.empty(3 * helper.npix, dtype=torch.float64, device=dev)
        wf.wf_alm2map(helper, T(P["a_signal"].ravel()), lmax, sig)
        helper.close()
        Nc = P["noise_cov"]
        N6 = np.stack([Nc[:, 0, 0], Nc[:, 1, 1], Nc[:, 2, 2], Nc[:, 0, 1], Nc[:, 0, 2], Nc[:, 1, 2]])
        common = {"noise_var": T(N6.ravel()), "mask": T(P["mask"]), "C_ell": T(P["c_ell"].T.ravel()),
                  "tol": args.pol_tol}
        nalm3 = 3 * (lmax + 1) * (lmax + 2) // 2
        items.append(dict(common, kind="wf", d=sig + T(P["noise"].ravel()), s_out=torch.empty_like(sig),
                          alm_out=torch.empty(nalm3, dtype=torch.complex128, device=dev)))
        items.append(dict(common, kind="fluct", g1=T(P["g1"].ravel()), g2=T(P["g2"].ravel()),
                          s_out=torch.empty_like(sig)))
        geo += [(ns, lmax)] * 2
    prec = args.pol_precision
    plans = [wf.wf_plan_create("healpix", nside=ns, lmax=l, precision=prec, ncomp=3) for ns, l in geo]
    for pl in plans:
        wf.wf_set_options(pl, maxiter=args.pol_maxiter)
    stream = torch.cuda.current_stream()

    def one_by_one():
        reps = []
        for pl, it in zip(plans, items):
            if it["kind"] == "wf":
                reps.append(wf.wf_solve(pl, it["d"], it["noise_var"], it["mask"], it["C_ell"], it["tol"], it["s_out"]))
            else:
                reps.append(wf.wf_fluct(pl, it["noise_var"], it["mask"], it["C_ell"], it["g1"], it["g2"], it["tol"],
                                        it["s_out"]))
        return reps

    def batched():
        return wf.wf_solve_batch(plans, items)

    out = {}
    legs = (("batched", batched),) if args.pol_no_alone else (("one_by_one", one_by_one), ("batched", batched))
    for name, fn in legs:
        if args.warmup > 0:
            fn()  # warm
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ts = []
        for _ in range(max(1, args.steps)):
            e0.record(stream)
            reps = fn()
            e1.record(stream)
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        iters = sum(r["iters"] for r in reps)
        ms = float(np.median(ts))
        out[name] = {"ms": ms, "iters": iters, "crs_per_s": n / (ms / 1e3), "iters_per_s": iters / (ms / 1e3),
                     "converged": int(sum(r["converged"] for r in reps)), "launches": int(sum(r["launches"] for r in reps))}
    # convergence of the batched solves by nside (the FP64 operator's verdict for mixed plans)
    by_nside = {}
    for (ns_, _), r_ in zip(geo, reps):
        b_ = by_nside.setdefault(str(ns_), {"solves": 0, "converged": 0, "max_final_residual": 0.0, "iters": []})
        b_["solves"] += 1
        b_["converged"] += int(bool(r_["converged"]))
        b_["max_final_residual"] = max(b_["max_final_residual"], float(r_["final_residual"]))
        b_["iters"].append(int(r_["iters"]))
    for b_ in by_nside.values():
        b_["iters"] = {"min": min(b_["iters"]), "max": max(b_["iters"])}
    per_item = [{"nside": int(ns_), "kind": it_["kind"], "iters": int(r_["iters"]), "converged": bool(r_["converged"]),
                 "final_residual": float(r_["final_residual"]), "status": int(r_["status"])}
                for (ns_, _), it_, r_ in zip(geo, items, reps)]
    err = None
    if rank == 0 and not args.no_cpu:
        # error against the FP64 oracle: one Wiener-filter result per nside, its returned
        # (I, Q, U) map on sampled rings against the oracle's synthesis of its returned
        # (T, E, B) a_lm (the first ring, the last polar-cap ring, a belt ring, the equator)
        import oracle

        err = {}
        for ns_ in sorted(set(int(x) for x in nsides)):
            i_ = 2 * [int(x) for x in nsides].index(ns_)
            lm_ = 2 * ns_
            na_ = (lm_ + 1) * (lm_ + 2) // 2
            npx = 12 * ns_ * ns_
            a3 = items[i_]["alm_out"].cpu().numpy().reshape(3, na_)
            m3 = items[i_]["s_out"].cpu().numpy().reshape(3, npx)
            rings = [0, ns_ - 1, ns_ + 3, 2 * ns_ - 1]
            e_ = 0.0
            for r0 in rings:
                sl = ring_slices(ns_, [r0])[0]
                t_ref = oracle.synthesis(ns_, lm_, lm_, a3[0], rings=(r0, r0 + 1))[sl]
                q_ref, u_ref = oracle.synthesis_pol(ns_, lm_, lm_, a3[1], a3[2], rings=(r0, r0 + 1))
                for got, ref in ((m3[0][sl], t_ref), (m3[1][sl], q_ref[sl]), (m3[2][sl], u_ref[sl])):
                    e_ = max(e_, float(np.max(np.abs(got - ref)) / max(float(np.max(np.abs(ref))), 1e-300)))
            err[str(ns_)] = e_
        err = {"result_map_vs_oracle_synthesis_of_result_alm": err,
               "basis": "max |GPU - oracle| / max |oracle| per component on rings 0, nside - 1, nside + 3, "
                        "2 nside - 1 of one Wiener-filter result per nside: the returned (I, Q, U) map against "
                        "the oracle's FP64 synthesis of the returned (T, E, B) a_lm"}
    # kernel families of one full-band polarised iteration at the largest nside (profiled replay)
    nb = int(max(nsides))
    it = items[int(np.argmax(nsides)) * 2]
    pl = wf.wf_plan_create("healpix", nside=nb, lmax=2 * nb, precision=prec, ncomp=3)
    wf.wf_set_options(pl, profile=1, refine_sweeps=0)
    k = 6
    wf.wf_set_schedule(pl, [1.0] * k, [2 * nb] * k)
    rep = wf.wf_solve(pl, it["d"], it["noise_var"], it["mask"], it["C_ell"], 1e-30, it["s_out"], trace_cap=k)
    fam = {kname: v / k for kname, v in rep["kernel_ms"].items() if v > 0}
    iter_ms = float(np.median(rep["iter_ms_trace"][1:]))
    pl.close()
    res = {"metric": "batched polarised constrained realisations (WF + fluctuation pairs) per second",
           "unit": "CR/s", "value": out["batched"]["crs_per_s"], "n_gpus": 1, "higher_is_better": True,
           "maps": n, "nsides": [int(x) for x in nsides], "one_by_one": out.get("one_by_one"),
           "batched": out["batched"], "by_nside": by_nside, "per_item": per_item, "err_vs_oracle": err,
           "speedup": out["one_by_one"]["ms"] / out["batched"]["ms"] if "one_by_one" in out else None,
           "full_band_iteration": {"nside": nb, "lmax": 2 * nb, "ms": iter_ms, "families_ms": fam},
           "dtype": {"fp64": "f64", "mixed": "f32+f64", "tf32": "tf32x3+f32+f64", "bf16": "bf16x3+f32+f64"}[prec],
           "data": "synthetic",
           "config": {"workload": "batch_IQU_CR_nside" + "-".join(str(c) for c in choices), "precision": prec,
                      "tol": args.pol_tol, "maxiter": args.pol_maxiter,
                      "timing": "CUDA events around the whole call, median of --steps runs"}}
    for p_ in plans:
        p_.close()
    if rank == 0:
        print(json.dumps(res))
    return 0


# --------------------------------------------------------------------------
# the two smaller workloads: flat 128 x 128 and HEALPix nside 512, FP64
# --------------------------------------------------------------------------
def _pcts(x):
    x = np.asarray(x, dtype=np.float64)
    return {"p50": float(np.percentile(x, 50)), "p99": float(np.percentile(x, 99)), "n": int(x.size)}


def run_config1(args):
    """Flat 128 x 128 periodic grid, FP64, one map: the whole solve (cooling from lambda 100 to 1
    and lambda = 1 down to tol) is one cooperative launch.  A step is one solve."""
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    P = gen.config_flat_128(0)
    n = P["nx"]
    d_h = np.fft.irfft2(P["a_signal"], s=(n, n), norm="ortho") + P["noise"]  # data: signal map + noise
    T = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    d, nv, mk, S = T(d_h.ravel()), T(P["noise_var"].ravel()), T(P["mask"].ravel()), T(P["S"].ravel())
    plan = wf.wf_plan_create("flat", n=n)
    wf.wf_set_options(plan, maxiter=20000)
    s_out = torch.empty(n * n, dtype=torch.float64, device=dev)
    stream = torch.cuda.current_stream()
    for _ in range(max(3, args.warmup)):
        wf.wf_solve(plan, d, nv, mk, S, args.tol, s_out)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    step_ms, iters = [], []
    clocks = Clocks(0)
    clocks.start()
    for _ in range(args.steps):
        e0.record(stream)
        rep = wf.wf_solve(plan, d, nv, mk, S, args.tol, s_out, trace_cap=20000)
        e1.record(stream)
        torch.cuda.synchronize()
        step_ms.append(e0.elapsed_time(e1))
        iters.append(rep["iters"])
    ck = clocks.stop()
    us_it = [1e3 * t / k for t, k in zip(step_ms, iters)]
    out = {"metric": "flat 128x128 FP64 Wiener filter: microseconds per messenger iteration and time to tol",
           "value": float(np.median(us_it)), "unit": "us/iter", "n_gpus": 1, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": float(np.mean(step_ms)), "higher_is_better": False,
           "dtype": "f64", "data": "synthetic",
           "config": {"workload": "flat_128x128_fp64", "tol": args.tol, "l2": "whole problem in registers and L2"},
           "time_to_tol_ms": _pcts(step_ms), "iters_per_solve": int(iters[-1]), "converged": bool(rep["converged"]),
           "final_residual": float(rep["final_residual"]), "lambda_levels": int(rep["n_levels"]),
           "gpu_launches_per_solve": int(rep["launches"]), "clocks": ck}
    if not args.no_cpu:
        import oracle

        basis = oracle.FlatBasis(n, n)
        obs = P["mask"] > 0
        nu = np.where(obs, 1.0 / P["noise_var"], 0.0)
        tau = float(P["noise_var"][obs].min())
        t0 = time.perf_counter()
        ref = oracle.messenger_solve(basis, nu * d_h, nu, P["S"], tau, tol=args.tol, maxiter=20000)
        t_or = time.perf_counter() - t0
        out["cpu_baseline"] = {"value": 1e6 * t_or / ref["iters"], "unit": "us/iter", "cores": 1, "kind": "oracle",
                               "sample": "one full oracle solve (numpy FFTs, one thread): %d iterations in %.2f s"
                                         % (ref["iters"], t_or), "time_to_tol_s": t_or}
        out["err_vs_oracle"] = {"s_wf_max_rel": float(np.max(np.abs(s_out.cpu().numpy() - ref["s"].ravel())) /
                                                     np.max(np.abs(ref["s"]))),
                                "note": "GPU and oracle each run their own schedule to tol (no replay)"}
    plan.close()
    print(json.dumps(out))
    return 0


def run_config2(args):
    """HEALPix nside 512 / lmax 1024, 13' beam, |b| < 20 deg plus 500 disks of 0.6 deg, FP64: full
    solves to tol (a step is one solve), iterations/s, per-iteration p50/p99, and the same solve in
    mixed precision beside it."""
    import torch

    import paper_1210_4931_gb300 as wf

    wf.load()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    nside, lmax = 512, 1024
    P = gen.config_nside512(0)
    T = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    out = {"metric": "HEALPix nside 512 / lmax 1024 FP64 Wiener filter: time to tol and messenger iterations/s",
           "unit": "iter/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True,
           "dtype": "f64", "data": "synthetic",
           "config": {"workload": "healpix_T_nside512_lmax1024_fp64", "tol": args.tol, "maxiter": args.maxiter,
                      "l2": "inputs (75 MB) fit in L2"}}
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clocks = Clocks(0)
    # fp64: the FP64 pipe throughout; fp64_emulated: the same FP64 plan with its Legendre transforms in
    # double-float arithmetic on the FP32 pipe (about 48 significant bits; wf_options.fp64_emulation)
    for leg in ("fp64", "fp64_emulated", "mixed"):
        prec = "mixed" if leg == "mixed" else "fp64"
        plan = wf.wf_plan_create("healpix", nside=nside, lmax=lmax, precision=prec)
        if prec == "mixed":
            wf.wf_plan_autotune(plan)
        s_sig = torch.empty(plan.npix, dtype=torch.float64, device=dev)
        wf.wf_alm2map(plan, T(P["a_signal"]), lmax, s_sig)
        d = s_sig + T(P["noise"])
        nv, mk, cl = T(P["noise_var"]), T(P["mask"]), T(P["c_ell"])
        s_out = torch.empty(plan.npix, dtype=torch.float64, device=dev)
        wf.wf_set_options(plan, maxiter=args.maxiter, profile=1, fp64_emulation=1 if leg == "fp64_emulated" else 0)
        steps = args.steps if leg == "fp64" else max(1, args.steps)
        for _ in range(args.warmup if leg == "fp64" else 1):
            wf.wf_solve(plan, d, nv, mk, cl, args.tol, s_out)
        torch.cuda.synchronize()
        if leg == "fp64":
            clocks.start()
        step_ms, reps = [], []
        for _ in range(steps):
            e0.record(stream)
            reps.append(wf.wf_solve(plan, d, nv, mk, cl, args.tol, s_out, trace_cap=args.maxiter + 16))
            e1.record(stream)
            torch.cuda.synchronize()
            step_ms.append(e0.elapsed_time(e1))
        if leg == "fp64":
            out["clocks"] = clocks.stop()
        last = reps[-1]
        it_ms = np.concatenate([r["iter_ms_trace"] for r in reps])
        full = np.concatenate([(r["lambda_trace"] == 1.0) & (r["L_trace"] == lmax) for r in reps])
        rec = {"iters_per_s": float(sum(r["iters"] for r in reps) / (sum(step_ms) / 1e3)),
               "time_to_tol_s": _pcts(np.array(step_ms) / 1e3) if last["converged"] else None,
               "converged": bool(last["converged"]), "iters_per_solve": int(last["iters"]),
               "final_residual": float(last["final_residual"]), "chi2_over_ndof": float(last["chi2_over_ndof"]),
               "iter_ms_full_band": _pcts(it_ms[full]) if full.any() else None,
               "time_to_residual_s": time_to_residual(last), "ms_per_step": float(np.mean(step_ms))}
        if leg == "fp64_emulated":
            rec["max_rel_diff_vs_fp64_map"] = float(torch.max(torch.abs(s_out - s_fp64)) / torch.max(torch.abs(s_fp64)))
        if leg == "fp64":
            s_fp64 = s_out.clone()
        out[leg] = rec
        plan.close()
    out["value"] = out["fp64"]["iters_per_s"]
    out["ms_per_step"] = out["fp64"]["ms_per_step"]
    if not args.no_cpu:
        t_it, desc, thr, _ = oracle_iteration_sample(nside, lmax, n_rings=16, n_m=16)
        out["cpu_baseline"] = {"value": 1.0 / t_it, "unit": "iter/s", "cores": thr, "kind": "oracle", "sample": desc,
                               "time_to_tol_s_extrapolated": t_it * out["fp64"]["iters_per_solve"]}
    print(json.dumps(out))
    return 0


def main():
    args = parse()
    if args.tol is None:
        args.tol = 1e-6 if args.config == 1 else 1e-4
    if args.impl == "reference":
        return run_reference(args)
    if args.config == 1:
        return run_config1(args)
    if args.config == 2:
        return run_config2(args)
    if args.serve:
        return run_serve(args)
    if args.batch > 0:
        return run_batch(args)
    if args.columns > 0:
        return run_columns(args)
    if args.pol_batch > 0:
        return run_pol_batch(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
