"""Benchmark of JARQ layer refinement on one GB300 (or N, weak scaling).

One step = one ``jarq_refine_layer`` call refining the Llama-2-7B q_proj
layer (4096 x 4096, g = 128, 3-bit, RTN host, K = 10 iterations, early stop
off) from its host state: the whole hot path (once the target projection
P = W H and its folded form; per iteration the Gram matrices, right-hand
sides and joint scale solve, then the sweep, a product and a Babai step per
block of two groups).  Inputs are seeded synthetic tensors resident in HBM; the
working set per step (W 64 MB, P and the folded P 128 MB each, digit planes
448 MB) exceeds the 129 MB L2.

``value`` is weights refined per second over all ranks; ``e2e`` is the same
metric through the C ABI with host buffers (host-to-device and back inside
the timed region).  ``--impl reference`` times the float64 oracle (the
reference arm of this build) on the host cores.

The line printed is short (below 2600 characters, so that it survives a log
that keeps the end of a program's output): the main workload in full, of the
other workloads and legs the figures.  ``--details FILE`` writes the whole
record, with every kernel's roofline.
"""
from __future__ import annotations

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

METRIC = "JARQ refine s/layer & weights/s at 7B shapes; % of tensor/HBM roofline"
UNIT = "weights/s"
WORKLOAD = "llama2_7b_q_proj_4096x4096_g128_w3"
PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
SM_COUNT = 152
FP32_LANES_PER_SM = 128
SM_MAX_MHZ = 2070.0
DTYPE = "f32 (integer-digit fp16/bf16 tensor-core products with exact partial sums, double-float accumulation)"

# DRAM bytes (read + write) per launch from one ncu capture of the main
# workload (q_proj; other workloads report null; the sweep kernels' figures
# are those of the first block, with ncu's cache flush before each launch; the
# Hessian kernel has none at the bench's token count); the summary kept with
# the profiles gives the capture's command.  A figure is
# valid while the kernel's source file is unchanged (first 12 hex digits of
# its SHA-1); otherwise the bench reports null.
TRAFFIC = {
    "sweep_product": ("k_tc_target.cu", "7ff0bf5bd113", 42.495e6 + 0.005e6),
    "sweep_babai": ("k_babai.cu", "1f2c6eaf91b0", 19.161e6 + 0.002e6),
    "gram": ("k_tc_gram.cu", "040880dfa541", 140.947e6 + 22.452e6),
    "proj": ("k_tc_proj.cu", "7359153c6634", 1336.274e6 + 137.113e6),
    "ptilde": ("k_tc_proj.cu", "7359153c6634", 134.262e6 + 143.167e6 + 293.427e6 + 97.857e6),
    "rhs": ("k_tc_proj.cu", "7359153c6634", 151.546e6 + 0.272e6),
    "whw": ("k_tc_proj.cu", "7359153c6634", 201.340e6 + 0.220e6),
    "slice_rows": ("k_tc_proj.cu", "7359153c6634", 67.128e6 + 72.345e6),
    "scale_solve": ("k_solve.cu", "c4ababeb8bae", 35.323e6 + 0.0),
}
HESSIAN_WORKLOAD = "llama2_7b_attn_in_4096_n262144"


def traffic_for(kernel):
    import hashlib
    ent = TRAFFIC.get(kernel)
    if not ent:
        return None
    path = os.path.join(ROOT, "paper_2609_38599_gb300", "csrc", ent[0])
    try:
        sha = hashlib.sha1(open(path, "rb").read()).hexdigest()[:12]
    except OSError:
        return None
    return ent[2] if sha == ent[1] else None


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default=WORKLOAD)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-configs", action="store_true",
                    help="skip timing the other workloads (tiny, down_proj, gate_proj, block)")
    ap.add_argument("--main-only", action="store_true",
                    help="time the main workload only: no post-passes, other workloads, "
                         "extra legs, end-to-end pass or CPU baseline (profiling runs)")
    ap.add_argument("--tokens", type=int, default=None,
                    help="calibration tokens of the Hessian workload (default: 128 x 2048)")
    ap.add_argument("--details", default=None, metavar="FILE",
                    help="write the whole record (rooflines and kernel times of every workload) here")
    ap.add_argument("--cpu-seconds", type=float, default=12.0,
                    help="target CPU time of the oracle baseline sample")
    return ap.parse_args()


def peaks():
    try:
        with open(PEAKS_FILE) as fh:
            pk = json.load(fh)
        return pk, "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


# --------------------------------------------------------------------------
# clocks sampled during the timed region
# --------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200", "-i", str(self.gpu)], stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as fh:
            for line in fh:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    smax.append(float(parts[2]))
                except ValueError:
                    continue
                for nm, v in zip(names, parts[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(nm)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# --------------------------------------------------------------------------
# oracle timing (CPU baseline and reference arm)
# --------------------------------------------------------------------------

def oracle_rows_per_second(lay_np, K, target_s, max_rows=None):
    """Time the float64 oracle on a growing sample of rows until ~target_s."""
    from oracle import Options, prepare_hessian, refine_layer
    prep = prepare_hessian(lay_np.H, lay_np.g)
    rng = np.random.default_rng(0)
    n = 4
    total_t, total_rows = 0.0, 0
    while True:
        rows = np.sort(rng.choice(lay_np.dout, size=min(n, lay_np.dout), replace=False))
        t0 = time.perf_counter()
        refine_layer(prep, lay_np.W[rows], lay_np.S0[rows], lay_np.Q0[rows], lay_np.Z[rows],
                     lay_np.bits, Options(max_iters=K, early_stop=False))
        dt = time.perf_counter() - t0
        total_t += dt
        total_rows += len(rows)
        if total_t >= target_s or (max_rows and total_rows >= max_rows) or len(rows) >= lay_np.dout:
            break
        n = int(min(lay_np.dout, max(n * 2, n * (target_s - total_t) / max(dt, 1e-3))))
    return total_rows, total_t


def layer_to_numpy(lay):
    from synth import Layer
    return Layer(lay.name, lay.W.cpu().numpy(), lay.H.cpu().numpy(), lay.S0.cpu().numpy(),
                 lay.Q0.cpu().numpy(), lay.Z.cpu().numpy(), lay.bits, lay.g, lay.K)


def run_reference(args, rank, world):
    if rank != 0:
        return 0
    import torch
    from synth import config_layer
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    lay = layer_to_numpy(config_layer(args.workload, device=dev))
    K = lay.K
    per_step_rows = 4
    from oracle import Options, prepare_hessian, refine_layer
    prep = prepare_hessian(lay.H, lay.g)
    rng = np.random.default_rng(1)
    times = []
    for it in range(args.warmup + args.steps):
        rows = np.sort(rng.choice(lay.dout, size=per_step_rows, replace=False))
        t0 = time.perf_counter()
        refine_layer(prep, lay.W[rows], lay.S0[rows], lay.Q0[rows], lay.Z[rows], lay.bits,
                     Options(max_iters=K, early_stop=False))
        if it >= args.warmup:
            times.append(time.perf_counter() - t0)
    t = float(np.mean(times))
    value = per_step_rows * lay.din / t
    cores = os.cpu_count()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": t * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": config_dict(lay, note=f"oracle on {per_step_rows} sampled rows per step"),
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"{per_step_rows} of {lay.dout} rows per step, K={K}, full din"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


def config_dict(lay, note=None):
    MB = 1 << 20
    pd, dd = lay.dout * lay.din, ((lay.din + 127) // 128 * 128) ** 2
    c = {"workload": lay.name, "din": lay.din, "dout": lay.dout, "group_size": lay.g,
         "bits": lay.bits, "K": lay.K, "early_stop": False, "host": "RTN",
         "l2": f"inputs larger than L2 (per step: W {4 * pd // MB} MB, P and the folded P "
               f"{8 * pd // MB} MB each as float pairs, digit planes of H and of the folded "
               f"rows {28 * dd // MB} MB)"}
    if note:
        c["note"] = note
    return c


# --------------------------------------------------------------------------
# our arm
# --------------------------------------------------------------------------

def kernel_model(kernel, lay, nsplit_bytes=0):
    """Algorithmic work of one launch and the roofline that bounds the kernel.

    Contractions count one MMA of useful work (2 x M x N x K); the digit
    products they issue (4 digit planes for the phase target product and the
    Gram, 18 digit pairs for the target projection) are reported separately
    as ``issued``.  Babai counts its dense triangular back substitution,
    g^2 flops per (row, group); the folded projection one MMA of its
    block-diagonal product (2 x p x d x g; 21 digit pairs issued).
    Memory-bound kernels count the bytes they must move once.
    """
    p, d, g, G = lay.dout, lay.din, lay.g, lay.din // lay.g
    # the sweep's blocks of 256 columns: the average launch of a sweep
    launches = -(-d // 256)
    if kernel == "sweep_product":
        return dict(bound="tensor", work=2.0 * p * d * d / launches,
                    issued=4 * 2.0 * p * d * d / launches)
    if kernel == "sweep_babai":
        return dict(bound="alu", work=1.0 * g * d * p / launches)
    if kernel == "hr_full":
        return dict(bound="tensor", work=2.0 * p * d * d, issued=8 * 2.0 * p * d * d)
    if kernel == "gram":
        blocks = G * (G + 1) / 2
        return dict(bound="tensor", work=2.0 * p * g * g * blocks, issued=4 * 2.0 * p * g * g * blocks)
    if kernel == "ptilde":
        return dict(bound="tensor", work=2.0 * p * d * g, issued=21 * 2.0 * p * d * g)
    if kernel == "scale_solve":
        # Gram (f64), rhs (f64), wHw, L_prev and the scales in; scales and L out
        return dict(bound="hbm", work=p * (8.0 * G * G + 8 * G + 8 + 8 + 4 * G + 4 * G + 8))
    if kernel == "grad":
        return dict(bound="hbm", work=p * d * (4 + 4 + 1) + p * G * 8)
    if kernel == "proj":
        return dict(bound="tensor", work=2.0 * p * d * d, issued=18 * 2.0 * p * d * d)
    if kernel == "rhs":
        # codes + double-float projection in, rhs (f64) out
        return dict(bound="hbm", work=p * d * (1 + 4 + 4) + p * G * (4 + 8))
    if kernel == "whw":
        return dict(bound="hbm", work=p * d * (4 + 4 + 4) + p * 8)
    if kernel == "slice_rows":
        return dict(bound="hbm", work=p * d * (4 + 4 * 2) + p * G * 4)
    return None


def roofline_entry(kernel, stats, lay, pk, peak_kind):
    m = kernel_model(kernel, lay)
    if not m or not stats.get("launches"):
        return None
    avg_s = stats["total_ms"] / stats["launches"] / 1e3
    if m["bound"] == "tensor":
        achieved = m["work"] / avg_s / 1e12
        peak, unit = pk["bf16_tflops_sustained"], "TFLOP/s"
        note = f"bf16 dense, sustained ({peak_kind})"
    elif m["bound"] == "alu":
        achieved = m["work"] / avg_s / 1e12
        peak, unit = SM_COUNT * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12, "TFLOP/s"
        note = "fp32 FMA: 152 SMs x 128 lanes x 2 flop x 2070 MHz"
    else:
        achieved = m["work"] / avg_s / 1e9
        peak, unit = pk["hbm_gbs"], "GB/s"
        note = f"HBM copy bandwidth ({peak_kind})"
    e = {"kernel": kernel, "bound": m["bound"], "achieved": achieved, "peak": peak, "unit": unit,
         "frac": achieved / peak,
         "traffic": traffic_for(kernel) if lay.name == WORKLOAD else None,
         "avg_us": avg_s * 1e6,
         "peak_note": note}
    if "issued" in m:
        e["issued_frac"] = m["issued"] / avg_s / 1e12 / peak
    return e


def run_ours(args, rank, world):
    import torch
    from paper_2609_38599_gb300 import jarq
    from synth import config_layer

    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    # each rank refines its own layer of the same shape (rank 0: the named
    # layer): independent problems, weak scaling, no collective on the path
    lay = config_layer(args.workload, device=dev, seed_offset=rank)
    hess = jarq.prepare(lay.H, lay.g)
    opts = jarq.default_options(max_iters=lay.K, early_stop=0)
    S = lay.S0.clone()
    Q = lay.Q0.clone()

    def step():
        S.copy_(lay.S0)
        Q.copy_(lay.Q0)
        jarq.refine(hess, lay.W, S, Q, lay.Z, lay.bits, options=opts, collect_stats=False)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    gpu_index = vis.split(",")[local] if vis and vis.split(",")[0].isdigit() else local
    sampler = ClockSampler(gpu_index)
    n0 = jarq.launch_count()
    sampler.start()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        step()
    e1.record()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    clocks = sampler.stop()
    launches = jarq.launch_count() - n0
    ms = e0.elapsed_time(e1) / args.steps
    if dist:
        t = torch.tensor([ms], device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms = float(t.item())
    # per-kernel device time: the same K steps again with a CUDA event pair
    # around every library launch, on the stream the kernels run on
    jarq.profile_reset()
    jarq.profile_enable(True)
    for _ in range(args.steps):
        step()
    torch.cuda.synchronize()
    jarq.profile_enable(False)
    weights = lay.din * lay.dout
    value = world * weights / (ms / 1e3)
    kernels = {}
    for k in jarq.KERNELS:
        n, tot = jarq.profile_read(k)
        if n:
            kernels[k] = {"launches": n, "total_ms": tot, "avg_us": 1e3 * tot / n,
                          "share": None}
    tot_all = sum(v["total_ms"] for v in kernels.values()) or 1.0
    for v in kernels.values():
        v["share"] = v["total_ms"] / tot_all
    # roofline of every modelled kernel; `roofline` is the one with the largest share
    pk, peak_kind = peaks()
    roofs = {k: roofline_entry(k, v, lay, pk, peak_kind) for k, v in kernels.items()}
    roofs = {k: v for k, v in roofs.items() if v}
    dom = max(kernels, key=lambda k: kernels[k]["total_ms"]) if kernels else None
    roof = roofs.get(dom)
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "s_per_layer": ms / 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": DTYPE,
        "data": "synthetic (seeded Llama-2-7B-shaped layer, RTN host)",
        "config": config_dict(lay), "roofline": roof, "roofline_all": roofs,
        "gpu_launches": launches,
        "kernel_timing": "CUDA event pair around every library launch on its stream, in a second "
                         "pass of the same K steps (the value pass runs without them)",
        "launches_per_step": launches / args.steps, "clocks": clocks, "kernels": kernels,
    }
    # write-back post-passes on the refined layer (not part of the step): the
    # returned weights cast to float16, the packed codes, canonicalisation
    post = {}
    if rank == 0 and not args.main_only:
        pk2, _ = peaks()

        def timed(fn, reps=5):
            fn()
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(reps):
                fn()
            b.record()
            torch.cuda.synchronize()
            return a.elapsed_time(b) / reps

        n_el = lay.dout * lay.din
        G = lay.din // lay.g
        S2, Q2, Z2 = S.clone(), Q.clone(), lay.Z.clone()
        t_dq = timed(lambda: jarq.dequantize(S, Q, lay.Z, lay.g, lay.bits, "float16"))
        t_pk = timed(lambda: jarq.pack_codes(Q, lay.bits))
        t_cn = timed(lambda: jarq.canonicalize(S2, Q2, Z2, lay.g, lay.bits))
        for name, ms_, by in (("dequantize_f16", t_dq, n_el * (1 + 2) + lay.dout * G * 8),
                              ("pack_codes", t_pk, n_el * (1 + lay.bits / 8)),
                              ("canonicalize", t_cn, n_el * 2 + lay.dout * G * 16)):
            post[name] = {"ms": ms_, "bytes": by, "GB_s": by / (ms_ / 1e3) / 1e9,
                          "hbm_frac": by / (ms_ / 1e3) / 1e9 / pk2["hbm_gbs"],
                          "note": "includes the code validation pass and a synchronize"}
        line["postpass"] = post
    if rank == 0 and not args.no_configs and not args.main_only:
        line["configs"] = configs_leg(args, jarq, dev)
    if rank == 0 and not args.main_only:
        line["hessian"] = hessian_leg(args, jarq, dev)
        line["early_stop"] = early_stop_leg(args, jarq, dev, lay, hess, ms)
        line["mu_target"] = mu_target_leg(args, jarq, dev, lay.name)
        line["ablations"] = ablation_leg(args, jarq, dev, lay, hess, ms)
    # end to end through the C ABI with pinned host buffers
    if not args.main_only:
        pin = lambda t: t.cpu().pin_memory().numpy()
        Wh, S0h, Q0h, Zh = pin(lay.W), pin(lay.S0), pin(lay.Q0), pin(lay.Z)
        Sh = torch.empty_like(lay.S0, device="cpu").pin_memory().numpy()
        Qh = torch.empty_like(lay.Q0, device="cpu").pin_memory().numpy()
        times = []
        for it in range(args.warmup + args.steps):
            Sh[...] = S0h
            Qh[...] = Q0h
            t0 = time.perf_counter()
            jarq.refine(hess, Wh, Sh, Qh, Zh, lay.bits, options=opts, collect_stats=False)
            dt = time.perf_counter() - t0
            if it >= args.warmup:
                times.append(dt)
        e2e_s = float(np.mean(times))
        if dist:
            t = torch.tensor([e2e_s], device=dev)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            e2e_s = float(t.item())
        line["e2e"] = {"value": world * weights / e2e_s, "unit": UNIT,
                       "h2d_bytes_per_step": int(Wh.nbytes + S0h.nbytes + Q0h.nbytes + Zh.nbytes),
                       "d2h_bytes_per_step": int(Sh.nbytes + Qh.nbytes),
                       "ms_per_step": e2e_s * 1e3}
    if rank == 0 and world == 1 and not args.no_cpu_baseline and not args.main_only:
        lay_np = layer_to_numpy(lay)
        rows, t = oracle_rows_per_second(lay_np, lay.K, args.cpu_seconds)
        line["cpu_baseline"] = {"value": rows * lay.din / t, "unit": UNIT,
                                "cores": os.cpu_count(), "kind": "oracle",
                                "sample": f"{rows} of {lay.dout} rows, K={lay.K}, full din, "
                                          f"{t:.1f} s"}
    hess.close()
    if rank == 0:
        if args.details:
            with open(args.details, "w") as fh:
                json.dump(line, fh)
        print(json.dumps(short_line(line)))
    if dist:
        dist.destroy_process_group()
    return 0


def _digits(x):
    """Floats of a nested record to five significant digits."""
    if isinstance(x, float):
        return float(f"{x:.5g}")
    if isinstance(x, dict):
        return {k: _digits(v) for k, v in x.items()}
    if isinstance(x, (list, tuple)):
        return [_digits(v) for v in x]
    return x


def short_line(full):
    """The printed line: the whole record without the parts that only explain
    it, kernels as [launches, us a launch] and the other legs reduced to their
    figures."""
    drop = ("roofline_all", "kernel_timing", "kernels", "postpass", "configs", "hessian", "early_stop",
            "mu_target", "ablations")
    out = {k: v for k, v in full.items() if k not in drop}
    extra = {}
    if "kernels" in full:
        extra["kernels"] = {k: [v["launches"], v["avg_us"]] for k, v in full["kernels"].items()}
    if "postpass" in full:
        extra["postpass_ms"] = {k: v["ms"] for k, v in full["postpass"].items()}
    if "configs" in full:
        extra["configs_s"] = {k: v.get("s_per_layer", v.get("s_per_block")) for k, v in full["configs"].items()}
    if "hessian" in full:
        h = full["hessian"]
        extra["hessian"] = {"kernel_ms": h["kernel_ms"], "tokens_per_s": h["tokens_per_s"],
                            "frac": h["roofline"]["frac"]}
    pick = {"early_stop": ("s_per_layer", "iters_mean"), "mu_target": ("ms_per_layer_mu_0.5", "ms_per_layer_mu_1.0"),
            "ablations": ("gap_independent_pct_median", "gap_coordinate_pct_median", "probe_ms_per_group",
                          "joint_over_fixed_heldout_pct_median")}
    for leg, keys in pick.items():
        if leg in full:
            extra[leg] = {k: full[leg][k] for k in keys}
    return {**out, **_digits(extra)}


def flush_l2(buf):
    """Overwrite a buffer larger than the 129 MB L2 (between timed steps)."""
    buf.add_(1.0)


def per_kernel(jarq, fn, steps):
    """Launches and device milliseconds of every library kernel over `steps`
    calls of fn, from the library's CUDA event pair around each launch on
    its stream."""
    import torch
    jarq.profile_reset()
    jarq.profile_enable(True)
    for _ in range(steps):
        fn()
    torch.cuda.synchronize()
    jarq.profile_enable(False)
    out = {}
    for k in jarq.KERNELS:
        n, tot = jarq.profile_read(k)
        if n:
            out[k] = (n, tot)
    return out


def summarise_kernels(parts, pk, peak_kind):
    """Per-kernel shares and roofline fractions from [(layer, {kernel: (n,
    ms)})]: a kernel's algorithmic work is summed over the layers it ran on
    (each with its own shape), divided by its summed device time."""
    tot = {}
    work = {}
    for lay, ks in parts:
        for k, (n, ms) in ks.items():
            t = tot.setdefault(k, [0, 0.0])
            t[0] += n
            t[1] += ms
            m = kernel_model(k, lay)
            if m:
                w = work.setdefault(k, [m["bound"], 0.0, 0.0])
                w[1] += m["work"] * n
                w[2] += m.get("issued", m["work"]) * n
    all_ms = sum(v[1] for v in tot.values()) or 1.0
    kernels = {k: {"launches": v[0], "total_ms": v[1], "avg_us": 1e3 * v[1] / v[0],
                   "share": v[1] / all_ms} for k, v in tot.items()}
    roofs = {}
    for k, (bound, w, wi) in work.items():
        sec = tot[k][1] / 1e3
        if bound == "tensor":
            ach, peak, unit = w / sec / 1e12, pk["bf16_tflops_sustained"], "TFLOP/s"
        elif bound == "alu":
            ach = w / sec / 1e12
            peak, unit = SM_COUNT * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12, "TFLOP/s"
        else:
            ach, peak, unit = w / sec / 1e9, pk["hbm_gbs"], "GB/s"
        e = {"kernel": k, "bound": bound, "achieved": ach, "peak": peak, "unit": unit,
             "frac": ach / peak, "peak_note": f"{peak_kind}"}
        if bound == "tensor":
            e["issued_frac"] = wi / sec / 1e12 / peak
        roofs[k] = e
    dom = max(kernels, key=lambda k: kernels[k]["total_ms"]) if kernels else None
    return kernels, roofs, dom


def configs_leg(args, jarq, dev):
    """Every workload besides the headline one, each timed on its own: the
    tiny layer, the Llama-2-7B down_proj layer, the Llama-3-8B gate_proj
    layer (one jarq_refine_layer call per step, K as configured, early stop
    off) and the Llama-2-7B decoder block (its three Hessians prepared and
    its seven layers refined per step).  Each step is timed alone by CUDA
    events on the current stream, with a 256 MiB buffer overwritten between
    steps so that no step starts with the previous one's data in L2; the
    median step is reported.  Per-kernel shares and roofline fractions come
    from a second pass with the library's per-launch event pairs."""
    import torch
    from synth import block_layers, config_layer
    pk, peak_kind = peaks()
    flush = torch.zeros(64 << 20, device=dev)
    out = {}

    def median_ms(step, warmup, steps):
        for _ in range(warmup):
            step()
        torch.cuda.synchronize()
        ts = []
        for _ in range(steps):
            flush_l2(flush)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            step()
            b.record()
            torch.cuda.synchronize()
            ts.append(a.elapsed_time(b))
        return float(statistics.median(ts)), ts

    for name, steps in (("tiny_256x256_g64_w3", 20),
                        ("llama2_7b_down_proj_4096x11008_g128_w4", 5),
                        ("llama3_8b_gate_proj_14336x4096_g128_w3", 5)):
        lay = config_layer(name, device=dev)
        hess = jarq.prepare(lay.H, lay.g)
        opts = jarq.default_options(max_iters=lay.K, early_stop=0)
        S, Q = lay.S0.clone(), lay.Q0.clone()

        def step():
            S.copy_(lay.S0)
            Q.copy_(lay.Q0)
            jarq.refine(hess, lay.W, S, Q, lay.Z, lay.bits, options=opts, collect_stats=False)

        n0 = jarq.launch_count()
        ms, ts = median_ms(step, 3, steps)
        launches = (jarq.launch_count() - n0) / (3 + steps)
        kernels, roofs, dom = summarise_kernels([(lay, per_kernel(jarq, step, steps))], pk,
                                                peak_kind)
        out[name] = {"din": lay.din, "dout": lay.dout, "group_size": lay.g, "bits": lay.bits,
                     "K": lay.K, "s_per_layer": ms / 1e3,
                     "weights_per_s": lay.din * lay.dout / (ms / 1e3), "steps": steps,
                     "step_ms_min_max": [min(ts), max(ts)], "launches_per_step": launches,
                     "dominant": dom, "roofline": roofs.get(dom), "roofline_all": roofs,
                     "kernels": kernels}
        hess.close()
        del lay, S, Q, hess
        torch.cuda.empty_cache()

    hs, layers = block_layers(device=dev)
    states = [(lay.S0.clone(), lay.Q0.clone()) for _, lay in layers]
    prof = {}

    def block_step(profile=False):
        hess = {k: jarq.prepare(h, 128) for k, h in hs.items()}
        if profile:
            torch.cuda.synchronize()
        for idx, ((hkey, lay), (S, Q)) in enumerate(zip(layers, states)):
            S.copy_(lay.S0)
            Q.copy_(lay.Q0)
            opts = jarq.default_options(max_iters=lay.K, early_stop=0)
            run = lambda: jarq.refine(hess[hkey], lay.W, S, Q, lay.Z, lay.bits, options=opts,
                                      collect_stats=False)
            if profile:
                prof[idx] = (lay, per_kernel(jarq, run, 1))
            else:
                run()
        for h in hess.values():
            h.close()

    n0 = jarq.launch_count()
    ms, ts = median_ms(block_step, 3, 3)
    launches = (jarq.launch_count() - n0) / 6
    block_step(profile=True)
    kernels, roofs, dom = summarise_kernels(list(prof.values()), pk, peak_kind)
    weights = sum(lay.din * lay.dout for _, lay in layers)
    out["llama2_7b_block"] = {
        "layers": [lay.name for _, lay in layers], "group_size": 128, "bits": 3, "K": 10,
        "hessians_prepared_per_step": len(hs), "s_per_block": ms / 1e3,
        "weights_per_s": weights / (ms / 1e3), "steps": 3, "step_ms_min_max": [min(ts), max(ts)],
        "launches_per_step": launches, "dominant": dom, "roofline": roofs.get(dom),
        "roofline_all": roofs,
        "kernels": kernels,
        "kernels_note": "refinement calls only (the Hessian preparation is in s_per_block)"}
    del hs, layers, states, flush
    torch.cuda.empty_cache()
    return out


def hessian_leg(args, jarq, dev, standalone=False):
    """The calibration Hessian H = X^T X of the q/k/v/gate/up input of a
    Llama-2-7B block (d = 4096) over 128 x 2048 fp16 tokens, one
    ``jarq_accumulate_hessian`` call: the step before refinement.  Timed by
    the library's CUDA event pair on its stream (kernel) and around the call
    (which synchronises).  Algorithmic work counts each unordered feature
    pair once: n d (d + 1) flops; the kernel issues whole 256 x 256 tiles
    on and above the diagonal."""
    import torch
    from synth import ACT_CONFIGS, config_activations
    X = config_activations(HESSIAN_WORKLOAD, device=dev, tokens=args.tokens)
    n, d = X.shape
    H = torch.zeros(d, d, device=dev)
    for _ in range(max(3, args.warmup)):
        jarq.accumulate_hessian(X, H)
    torch.cuda.synchronize()
    reps = max(1, args.steps) if standalone else 5
    jarq.profile_reset()
    jarq.profile_enable(True)
    t0 = time.perf_counter()
    for _ in range(reps):
        jarq.accumulate_hessian(X, H)
    call_ms = (time.perf_counter() - t0) / reps * 1e3
    jarq.profile_enable(False)
    nl, tot = jarq.profile_read("syrk")
    k_ms = tot / max(1, nl)
    pk, peak_kind = peaks()
    work = float(n) * d * (d + 1)
    ct = (d + 255) // 256
    issued = ct * (ct + 1) // 2 * 2.0 * 256 * 256 * (-(-n // 64) * 64)
    achieved = work / (k_ms / 1e3) / 1e12
    peak = pk["bf16_tflops"]
    out = {"workload": HESSIAN_WORKLOAD, "tokens": n, "din": d, "call_ms": call_ms,
           "kernel_ms": k_ms, "tokens_per_s": n / (k_ms / 1e3),
           "roofline": {"kernel": "syrk", "bound": "tensor", "achieved": achieved, "peak": peak,
                        "unit": "TFLOP/s", "frac": achieved / peak,
                        "issued_frac": issued / (k_ms / 1e3) / 1e12 / peak,
                        "traffic": traffic_for("syrk"),
                        "peak_note": f"fp16 dense = bf16 dense rate, burst ({peak_kind})"},
           "l2": f"X is {n * d * 2 / 2**20:.0f} MiB, larger than the 129 MB L2",
           "data": "synthetic fp16 activations (rank-64 correlated + outlier channels)"}
    del X, H
    torch.cuda.empty_cache()
    if not args.no_cpu_baseline:
        from oracle import accumulate_hessian
        from synth import activations_np
        c = ACT_CONFIGS[HESSIAN_WORKLOAD]
        ns = 4096
        Xs = activations_np(ns, d, rank=c["rank"], n_out=c["n_out"], out_scale=c["out_scale"],
                            D_lo=c["D_lo"], seed=c["seed"])
        t0 = time.perf_counter()
        accumulate_hessian(Xs)
        t = time.perf_counter() - t0
        out["cpu_baseline"] = {"value": ns / t, "unit": "tokens/s", "cores": os.cpu_count(),
                               "kind": "oracle",
                               "sample": f"{ns} of {n} tokens, d={d}, float64, {t:.2f} s"}
    return out


def ablation_leg(args, jarq, dev, lay, hess, joint_ms):
    """Tab. mechanism-summary (a) on the bench layer, from its RTN host
    state (App. "Refinement Mechanisms"):
    * scale fits with the host codes: median over rows of the gap
      100 (F_method - F_joint) / F_host of the independent fit and of 3-pass
      coordinate descent, and the call times;
    * multi-code probe of every (row, group): share of cases where one Babai
      proposal still lowers F after single-code search stops, median codes
      such a proposal changes;
    * Fixed (host scales, code sweeps) against Joint at equal time: Joint is
      the timed K = 10 step; Fixed gets the sweeps that fit in that time; both
      final states are scored on a held-out Hessian (the same distribution,
      other tokens): median over rows of 100 (F_fixed - F_joint) / F_fixed and
      the share of rows Joint improves."""
    import torch
    from synth import CONFIGS
    from synth.layers import hessian_torch
    out = {}
    ev = lambda: (torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))

    def timed(fn):
        fn()
        torch.cuda.synchronize()
        a, b = ev()
        a.record()
        r = fn()
        b.record()
        torch.cuda.synchronize()
        return r, a.elapsed_time(b)

    F = {}
    tms = {}
    for m in ("joint", "independent", "coordinate"):
        S = lay.S0.clone()
        (Fb, Fa), tms[m] = timed(lambda: jarq.fit_scales(hess, lay.W, S.copy_(lay.S0), lay.Q0,
                                                         lay.Z, lay.bits, m, 3))
        F[m], F["host"] = Fa.cpu().numpy(), Fb.cpu().numpy()
    for m in ("independent", "coordinate"):
        out[f"gap_{m}_pct_median"] = float(np.median(100.0 * (F[m] - F["joint"]) / F["host"]))
    out["fit_ms"] = tms
    out["coordinate_time_ratio"] = tms["coordinate"] / tms["joint"]
    G = lay.din // lay.g
    acc, chg, moves = [], [], []
    t0 = time.perf_counter()
    for i in range(G):
        r = jarq.multicode_probe(hess, lay.W, lay.S0, lay.Q0, lay.Z, lay.bits, i)
        a = r["accepted"].cpu().numpy().astype(bool)
        acc.append(a)
        chg.append(r["changed"].cpu().numpy()[a])
        moves.append(r["moves"].cpu().numpy())
    out["probe_ms_per_group"] = (time.perf_counter() - t0) / G * 1e3
    acc = np.concatenate(acc)
    chg = np.concatenate(chg)
    out["babai_after_single_code_pct"] = 100.0 * float(acc.mean())
    out["median_codes_changed"] = float(np.median(chg)) if chg.size else 0.0
    out["median_single_code_moves"] = float(np.median(np.concatenate(moves)))
    # Fixed vs Joint at equal time
    S, Q = lay.S0.clone(), lay.Q0.clone()
    o = jarq.default_options(max_iters=lay.K, early_stop=0)
    o.fixed_grid = 1

    def fixed(k):
        o.max_iters = k
        S.copy_(lay.S0)
        Q.copy_(lay.Q0)
        jarq.refine(hess, lay.W, S, Q, lay.Z, lay.bits, options=o, collect_stats=False)

    _, t_fix = timed(lambda: fixed(lay.K))
    k_fixed = max(1, int(lay.K * joint_ms / t_fix))
    fixed(k_fixed)
    torch.cuda.synchronize()
    Sf, Qf = S.clone(), Q.clone()
    Sj, Qj = lay.S0.clone(), lay.Q0.clone()
    jarq.refine(hess, lay.W, Sj, Qj, lay.Z, lay.bits, max_iters=lay.K, early_stop=0,
                collect_stats=False)
    c = CONFIGS[lay.name]
    H_ho = hessian_torch(c["din"], c["rank"], c["n_out"], c["out_scale"], c["tokens"] // 4,
                         c["D_lo"], c["seed"], dev, token_seed=9000 + c["seed"])
    h_ho = jarq.prepare(H_ho, lay.g)
    Ff = jarq.objective(h_ho, lay.W, Sf, Qf, lay.Z, lay.bits).cpu().numpy()
    Fj = jarq.objective(h_ho, lay.W, Sj, Qj, lay.Z, lay.bits).cpu().numpy()
    h_ho.close()
    out["fixed_sweeps_in_joint_time"] = k_fixed
    out["joint_over_fixed_heldout_pct_median"] = float(np.median(100.0 * (Ff - Fj) / Ff))
    out["rows_improved_by_joint"] = float(np.mean(Fj < Ff))
    out["heldout"] = f"{c['tokens'] // 4} other tokens of the same distribution"
    return out


def early_stop_leg(args, jarq, dev, lay, hess, fixed_ms):
    """The main layer with the early stop of App. E (Eq. strict_stopping,
    default thresholds) against the fixed K-iteration run of the main line:
    seconds per layer, the rows' last solved iteration and, per iteration k,
    the share of rows and of the pairs of row tiles (256 rows) still solved at
    k (a pair whose rows have all stopped skips its products and Gram blocks;
    stopped rows skip the scale solve and the Babai step)."""
    import torch
    opts = jarq.default_options(max_iters=lay.K, early_stop=1)
    S = lay.S0.clone()
    Q = lay.Q0.clone()

    def step():
        S.copy_(lay.S0)
        Q.copy_(lay.Q0)
        jarq.refine(hess, lay.W, S, Q, lay.Z, lay.bits, options=opts, collect_stats=False)

    for _ in range(2):
        step()
    torch.cuda.synchronize()
    steps = max(3, args.steps // 2)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    n0 = jarq.launch_count()
    a.record()
    for _ in range(steps):
        step()
    b.record()
    torch.cuda.synchronize()
    ms = a.elapsed_time(b) / steps
    launches = (jarq.launch_count() - n0) / steps
    S.copy_(lay.S0)
    Q.copy_(lay.Q0)
    st = jarq.refine(hess, lay.W, S, Q, lay.Z, lay.bits, options=opts, collect_stats=True)
    it = st.iters.cpu().numpy().astype(np.int64)
    ntile = (len(it) + 255) // 256
    tile_max = np.zeros(ntile * 256, np.int64)
    tile_max[:len(it)] = it
    tile_max = tile_max.reshape(ntile, 256).max(axis=1)
    K = lay.K
    return {"K": K, "tau_rel": opts.tau_rel, "tau_abs": opts.tau_abs, "steps": steps,
            "s_per_layer": ms / 1e3, "weights_per_s": lay.din * lay.dout / (ms / 1e3),
            "fixed_K_s_per_layer": fixed_ms / 1e3, "speedup_vs_fixed": fixed_ms / ms,
            "launches_per_step": launches, "iters_mean": float(it.mean()),
            "iters_hist": np.bincount(it, minlength=K + 1).tolist(),
            "rows_solved_at_k": [float(np.mean(it >= k)) for k in range(1, K + 1)],
            "tiles_solved_at_k": [float(np.mean(tile_max >= k)) for k in range(1, K + 1)]}


def mu_target_leg(args, jarq, dev, name):
    """The same layer shape refined on the propagation-corrected target
    (mu = 0.5; H, K = X~^T X and XX = X^T X from 128 x 2048 drifted fp16
    tokens) against the main target (mu = 1) on the same H: per-layer time
    of each, CUDA events on the launching stream, five timed calls after
    three warm-up calls."""
    import torch
    from synth.qep import mu_config_layer
    lay, K, XX, nu2 = mu_config_layer(name, device=dev)
    hess = jarq.prepare(lay.H, lay.g)
    opts = jarq.default_options(max_iters=lay.K, early_stop=0)
    S, Q = lay.S0.clone(), lay.Q0.clone()

    def run(mu):
        S.copy_(lay.S0)
        Q.copy_(lay.Q0)
        jarq.refine_mu(hess, lay.W, S, Q, lay.Z, lay.bits, K, XX, mu, nu2, options=opts,
                       collect_stats=False)

    out = {}
    for mu in (0.5, 1.0):
        for _ in range(3):
            run(mu)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            run(mu)
        b.record()
        torch.cuda.synchronize()
        out[f"ms_per_layer_mu_{mu}"] = a.elapsed_time(b) / 5
    out["extra_ms"] = out["ms_per_layer_mu_0.5"] - out["ms_per_layer_mu_1.0"]
    out["weights_per_s_mu_0.5"] = lay.din * lay.dout / (out["ms_per_layer_mu_0.5"] / 1e3)
    out["workload"] = name + " on the mu = 0.5 target (drift 0.05)"
    hess.close()
    del lay, K, XX
    torch.cuda.empty_cache()
    return out


def run_hessian(args, rank, world):
    """``--workload llama2_7b_attn_in_4096_n262144``: the Hessian step alone,
    one line of its own (tokens/s)."""
    import torch
    from paper_2609_38599_gb300 import jarq
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    n0 = jarq.launch_count()
    h = hessian_leg(args, jarq, dev, standalone=True)
    line = {"metric": "calibration Hessian X^T X, tokens/s", "value": world * h["tokens_per_s"],
            "unit": "tokens/s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": h["kernel_ms"], "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "fp16 products, f32 sums", "data": h["data"],
            "config": {"workload": HESSIAN_WORKLOAD, "tokens": h["tokens"], "din": h["din"],
                       "l2": h["l2"]},
            "roofline": h["roofline"], "gpu_launches": jarq.launch_count() - n0,
            "call_ms": h["call_ms"]}
    if "cpu_baseline" in h:
        line["cpu_baseline"] = h["cpu_baseline"]
    if rank == 0:
        print(json.dumps(line))
    return 0


BLOCK_WORKLOAD = "llama2_7b_block"


def run_block(args, rank, world):
    """The Llama-2-7B decoder block, timed end to end per block: the three
    Hessians prepared and the seven layers refined (K = 10 each) per step."""
    import torch
    from paper_2609_38599_gb300 import jarq
    from synth import block_layers

    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    hs, layers = block_layers(device=dev)
    states = [(lay.S0.clone(), lay.Q0.clone()) for _, lay in layers]

    def step():
        hess = {k: jarq.prepare(h, 128) for k, h in hs.items()}
        for (hkey, lay), (S, Q) in zip(layers, states):
            S.copy_(lay.S0)
            Q.copy_(lay.Q0)
            opts = jarq.default_options(max_iters=lay.K, early_stop=0)
            jarq.refine(hess[hkey], lay.W, S, Q, lay.Z, lay.bits, options=opts, collect_stats=False)
        for h in hess.values():
            h.close()

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    gpu_index = vis.split(",")[local] if vis and vis.split(",")[0].isdigit() else local
    sampler = ClockSampler(gpu_index)
    n0 = jarq.launch_count()
    sampler.start()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        step()
    e1.record()
    torch.cuda.synchronize()
    clocks = sampler.stop()
    launches = jarq.launch_count() - n0
    ms = e0.elapsed_time(e1) / args.steps
    weights = sum(lay.din * lay.dout for _, lay in layers)
    line = {
        "metric": METRIC, "value": world * weights / (ms / 1e3), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "s_per_block": ms / 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": DTYPE,
        "data": "synthetic (seeded Llama-2-7B-shaped block, RTN host)",
        "config": {"workload": BLOCK_WORKLOAD, "layers": [lay.name for _, lay in layers],
                   "group_size": 128, "bits": 3, "K": 10, "early_stop": False,
                   "hessians_prepared_per_step": len(hs),
                   "l2": "inputs larger than L2 (H of down_proj alone 485 MB)"},
        "roofline": None, "gpu_launches": launches,
        "launches_per_step": launches / args.steps, "clocks": clocks,
    }
    if rank == 0:
        print(json.dumps(line))
    return 0


def main():
    args = parse_args()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if args.impl == "reference":
        return run_reference(args, rank, world)
    if args.workload == BLOCK_WORKLOAD:
        return run_block(args, rank, world)
    if args.workload == HESSIAN_WORKLOAD:
        return run_hessian(args, rank, world)
    return run_ours(args, rank, world)


if __name__ == "__main__":
    sys.exit(main())
