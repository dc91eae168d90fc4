#!/usr/bin/env python
"""Throughput of the micromagnetic hot path on one GB300 (or N independent replicas).

Workload (default): the 512 x 512 x 16 permalloy film with 2 nm cells
(padded FFT grid 1024 x 1024 x 32), Ms = 8e5 A/m, A = 1.3e-11 J/m,
alpha = 0.5, a seeded vortex with 5 % noise, relaxed with adaptive RKF45
(tol 1e-5) through the library's relax() entry point.  One step = one
accepted RKF45 step of relax(): six stages, each a full demag + exchange
field evaluation fused with the LLG right-hand side, the device-side step
controller, and relax()'s torque check every ten trials.

Reported: field evals/s (one demag + exchange evaluation of the whole mesh)
as ``value``, LLG Mcell-steps/s, the roofline of the dominant kernel (its
launches timed with CUDA events on the library's stream inside the timed
region), clocks sampled during the timed region, an end-to-end number
through the public API with host buffers, and the CPU oracle timed on a
bounded sample.  ``--impl reference`` times the oracle instead.

Multi-GPU (torchrun): the method runs on one GPU; N ranks run N independent
replicas (one per GPU, no data exchange) and ``value`` sums their work over
the slowest rank's time.
"""

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import workloads as wl  # noqa: E402

METRIC = "demag+exch field evals/s & LLG Mcell-steps/s, % HBM roofline, vs FP64 oracle"
UNIT = "field evals/s"
FALLBACK_HBM_GBS = 6800.0


def parse():
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=60)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--precision", choices=["f32", "f64"], default="f32")
    ap.add_argument("--fft-mode", choices=["fp32", "tf32", "bf16", "ff", "f4"], default="fp32",
                    help="tf32/bf16: tensor-core split-precision y passes (f32); ff: float-float demag passes (f64); "
                         "f4: y forward, z product and y inverse fused over kx planes in 4-CTA clusters (f32)")
    ap.add_argument("--workload", choices=["film512"], default="film512")
    ap.add_argument("--solver", choices=["relax", "bb"], default="relax",
                    help="relax: adaptive RKF45 (default); bb: Barzilai-Borwein minimiser iterations")
    ap.add_argument("--dmi", type=float, default=0.0, help="interfacial DMI constant D in J/m^2 (0: off)")
    ap.add_argument("--stt", type=float, default=0.0,
                    help="Slonczewski current density J in A/m^2 (0: off; P 0.4, Lambda 2, p along z)")
    ap.add_argument("--e2e-steps", type=int, default=10)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the FP64 sub-line, the cuFFT comparison, the ALU roofs and the window statistics")
    ap.add_argument("--relax-to", type=float, default=0.0, metavar="T",
                    help="relax the film to simulated time T (s) in one relax() call and report that run")
    ap.add_argument("--cpu-budget", type=float, default=150.0, help="seconds of oracle work for the reference arm")
    ap.add_argument("--per-field", type=int, default=0, metavar="ITERS",
                    help="time mm_demag_field and mm_exchange_field alone, the paper's per-field protocol "
                         "(1000 warm-ups, then ITERS timed calls each, e.g. 10000) and exit")
    ap.add_argument("--ingest-ncu", metavar="CSV", default=None,
                    help="write profiles/traffic.json from an ncu raw CSV export and exit")
    return ap.parse_args()


# ---------------------------------------------------------------- helpers
def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def reduce_over_ranks(dist, ms, evals, accepted, device):
    """Replicas: the slowest rank's timed region and the work of all ranks,
    (max ms, sum of field evaluations, sum of accepted steps)."""
    if dist is None:
        return ms, float(evals), float(accepted)
    import torch
    t = torch.tensor([ms, float(evals), float(accepted)], dtype=torch.float64, device=device)
    mx = t.clone()
    dist.all_reduce(mx, op=dist.ReduceOp.MAX)
    sm = t.clone()
    dist.all_reduce(sm, op=dist.ReduceOp.SUM)
    return float(mx[0]), float(sm[1]), float(sm[2])


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


# the sources each timed kernel family is compiled from: stored ncu traffic
# stays valid while these files are unchanged
KERNEL_SOURCES = {
    "demag": ("mm_demag.cu", "mm_zline.cu", "mm_plane_launch.cuh", "mm_plane.cuh", "mm_fft.cuh", "mm_regfft.cuh",
              "mm_ff.cuh", "mm_tma.cuh", "mm_tcgen05.cuh", "mm_internal.cuh"),
    "stage": ("mm_llg.cu", "mm_fields.cuh", "mm_rk.cuh", "mm_ff.cuh", "mm_internal.cuh"),
}
FAMILY = {"xfwd": "demag", "yfwd": "demag", "zconv": "demag", "yinv": "demag", "xinv": "demag", "stage": "stage"}
# kernel-name prefixes of each timed class as ncu reports them
NCU_NAMES = {"xfwd": "k_xfwd", "yfwd": "k_cols", "yinv": "k_cols", "zconv": ("k_zconv", "k_zline"), "xinv": "k_xinv",
             "stage": "k_stage"}


def source_hash(kernel):
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2606_01114_gb300", "csrc")
    for fn in KERNEL_SOURCES[FAMILY[kernel]]:
        with open(os.path.join(csrc, fn), "rb") as f:
            h.update(fn.encode())
            h.update(f.read())
    return h.hexdigest()[:16]


def traffic_key(precision, fft_mode):
    """The name under which a mode's captures are stored: the plain passes
    under the precision, any other mode (kernels of its own) under its name."""
    return precision if fft_mode == "fp32" else fft_mode


def ncu_traffic(kernel, precision):
    """DRAM bytes per launch of ``kernel`` from the committed ncu summary, or
    None when the kernel's sources changed since the counters were taken."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            t = json.load(f)
    except Exception:
        return None
    e = t.get(f"{kernel}/{precision}")
    if not e or e.get("source_sha") != source_hash(kernel):
        return None
    return float(e["bytes_per_launch"])


# a kernel's name in an ncu export, with its template arguments when it has any
KNAME = r"(k_\w+)(?:<([^>]*)>)?\("


def ingest_ncu(csv_path, precision, workload):
    """Update profiles/traffic.json from an ncu raw CSV export
    (``ncu -i rep --page raw --csv``): per timed kernel class found in the
    capture, the dram__bytes_read.sum + dram__bytes_write.sum of its first
    captured launch (for the y passes, the forward launch is the one whose
    name carries DIR = -1), stamped with the current source hash of its
    family; classes not in the capture keep their entries."""
    import csv
    import re
    with open(csv_path, newline="") as f:
        rows = list(csv.reader(f))
    head = rows[0]
    col = {name: head.index(name) for name in ("Kernel Name", "dram__bytes_read.sum", "dram__bytes_write.sum")}
    units = rows[1] if len(rows) > 1 and not rows[1][col["Kernel Name"]] else None
    data = rows[2:] if units else rows[1:]
    scale = {"byte": 1, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9}

    def to_bytes(r, metric):
        unit = units[col[metric]] if units else "byte"
        return float(r[col[metric]].replace(",", "")) * scale.get(unit, 1)

    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            out = json.load(f)          # kernels absent from this capture keep their entries
    except Exception:
        out = {}
    out["_note"] = ("DRAM bytes per launch (dram__bytes_read.sum + dram__bytes_write.sum) from an ncu "
                    "capture; valid while the kernel family's sources hash to source_sha")
    for k, prefix in NCU_NAMES.items():
        if k == "stage":
            # the byte model is the average over the RKF45 stages: average the captured stage launches
            got = [r for r in data if (lambda mt: mt and mt.group(1).startswith(prefix))(
                re.search(KNAME, r[col["Kernel Name"]]))]
            if got:
                rd = sum(to_bytes(r, "dram__bytes_read.sum") for r in got) / len(got)
                wr = sum(to_bytes(r, "dram__bytes_write.sum") for r in got) / len(got)
                name = re.search(KNAME, got[0][col["Kernel Name"]]).group(1)
                out[f"{k}/{precision}"] = {"kernel": f"{name} (average of {len(got)} stage launches)",
                                           "workload": workload, "bytes_per_launch": int(rd + wr), "read": int(rd),
                                           "write": int(wr), "source_sha": source_hash(k)}
            continue
        for r in data:
            mt = re.search(KNAME, r[col["Kernel Name"]])
            if not mt or not mt.group(1).startswith(prefix):
                continue
            targs = mt.group(2) or ""
            if k in ("yfwd", "yinv"):
                # k_cols_reg / k_cols_tma<L1, L2, DIR, PIN, POUT>: DIR is the third argument
                direction = int(targs.split(",")[2].replace("(int)", "").strip())
                if (direction < 0) != (k == "yfwd"):
                    continue
            rd, wr = to_bytes(r, "dram__bytes_read.sum"), to_bytes(r, "dram__bytes_write.sum")
            out[f"{k}/{precision}"] = {"kernel": mt.group(1) + (f"<{targs}>" if mt.group(2) is not None else ""),
                                       "workload": workload,
                                       "bytes_per_launch": int(rd + wr), "read": int(rd), "write": int(wr),
                                       "source_sha": source_hash(k)}
            break
    with open(path, "w") as f:
        json.dump(out, f, indent=1)
    print(json.dumps(out, indent=1))
    return 0


class ClockSampler:
    """nvidia-smi samples every 200 ms while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
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
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# GB300 FP64 rate: 152 SMs x 2 FP64 FMA / clock x 2 flop x 2.07 GHz = 1.26 TFLOP/s,
# the 1.25 TFLOP/s nominal figure of the part; no FP64 peak is measured here
FP64_TFLOPS = 1.25


def algorithmic_flops(kind, n):
    """Floating-point operations of one launch (FP64 roofline).  A complex
    FFT of length L counts 5 L log2 L; the z pass adds the 3 x 3 real-tensor
    product (30 flops per k point) to its 3 forward and 3 inverse transforms;
    the x passes add the real-to-complex unpacking (10 flops per kept
    frequency)."""
    import math
    nx, ny, nz = n
    Hx = nx + 1 if nx > 1 else 1
    Py = 2 * ny if ny > 1 else 1
    Pz = 2 * nz if nz > 1 else 1

    def fft(L):
        return 5.0 * L * math.log2(L) if L > 1 else 0.0
    xrows = 3 * nz * ny
    return {
        "xfwd": xrows * (fft(nx) + 10.0 * Hx),
        "xinv": xrows * (fft(nx) + 10.0 * Hx),
        "yfwd": 3 * nz * Hx * fft(Py),
        "yinv": 3 * nz * Hx * fft(Py),
        "zconv": Py * Hx * (6 * fft(Pz) + 30.0 * Pz),
    }.get(kind)


def algorithmic_bytes(kind, n, s, Ms_cell=False):
    """Bytes one launch of kernel class ``kind`` must move (s = element size).

    Demag passes (Hx = nx+1 kept x frequencies, Py = 2 ny, Pz = 2 nz):
      xfwd  reads M (3 N s), writes 3 nz ny Hx complex
      yfwd  reads 3 nz ny Hx, writes 3 nz Py Hx complex
      zconv reads and writes 3 nz Py Hx complex, reads the kernel octant
            6 (Pz/2+1)(Py/2+1) Hx reals
      yinv  mirror of yfwd;  xinv mirror of xfwd
    RKF45 stage (average of its six launches): 42 vector fields of 3 N s
    in total per step (m_in, H_d, m0, the stage slopes the tableau needs,
    k_s and the next trial state)."""
    nx, ny, nz = n
    N = nx * ny * nz
    Hx = nx + 1 if nx > 1 else 1
    Py = 2 * ny if ny > 1 else 1
    Pz = 2 * nz if nz > 1 else 1
    c = 2 * s
    small = 3 * nz * ny * Hx * c
    big = 3 * nz * Py * Hx * c
    vec = 3 * N * s
    ms = N * s if Ms_cell else 0
    return {
        "xfwd": vec + ms + small,
        "yfwd": small + big,
        "zconv": 2 * big + 6 * (Pz // 2 + 1) * (Py // 2 + 1) * Hx * s,
        "yinv": small + big,
        "xinv": small + vec,
        "stage": 42 * vec / 6.0,
    }.get(kind)


# ------------------------------------------------------------ CPU oracle
class ThreadedFFT:
    """rfftn / irfftn of scipy.fft on ``workers`` threads: the same real
    transforms the oracle takes from numpy, spread over the host's cores
    (used only to time the oracle; its arithmetic is unchanged)."""

    def __init__(self, workers):
        import scipy.fft
        self._f = scipy.fft
        self.workers = workers

    def rfftn(self, a, s=None, axes=None):
        return self._f.rfftn(a, s=s, axes=axes, workers=self.workers)

    def irfftn(self, a, s=None, axes=None):
        return self._f.irfftn(a, s=s, axes=axes, workers=self.workers)


def host_cpu():
    """(logical cores, CPU model) of this host."""
    model = "unknown"
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for ln in out.splitlines():
            if ln.startswith("Model name:"):
                model = ln.split(":", 1)[1].strip()
                break
    except Exception:
        pass
    return os.cpu_count() or 1, model


def oracle_setup(w, workers):
    from oracle import micromag
    t0 = time.perf_counter()
    p = micromag.Problem(w["n"], w["d"], Ms=w["Ms"], A=w["A"], alpha=w["alpha"])
    if workers > 1:
        p.fft = ThreadedFFT(workers)
    nh = p.kernel_hat()
    p.kernel_hat = lambda: nh          # keep the transformed kernel (setup, not timed)
    p._kernel = None
    return p, time.perf_counter() - t0


def oracle_field_eval(p, m):
    return p.demag_fft(m) + p.exchange(m)


def time_oracle(p, m, evals):
    t0 = time.perf_counter()
    for _ in range(evals):
        oracle_field_eval(p, m)
    return (time.perf_counter() - t0) / evals


def cpu_baseline(w, m):
    """The oracle's field evaluation timed on all host cores (threaded FFT)
    and on one thread (numpy's FFT), one evaluation each after a warm-up."""
    cores, model = host_cpu()
    n = w["n"]
    ncell = n[0] * n[1] * n[2]
    p, setup_s = oracle_setup(w, cores)
    oracle_field_eval(p, m)
    t_all = time_oracle(p, m, 2)
    p.fft = __import__("numpy").fft
    t_one = time_oracle(p, m, 1)
    return {"value": 1.0 / t_all, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": (f"demag + exchange field evaluations of the {n[0]}x{n[1]}x{n[2]} film, float64 numpy with "
                       f"scipy.fft on {cores} threads ({model}), mean of 2 after 1 warm-up: {t_all:.2f} s each; "
                       f"Newell kernel setup ({setup_s:.0f} s) excluded"),
            "llg_mcell_steps_per_s": (1.0 / t_all) / 6.0 * ncell / 1e6,
            "cpu_model": model,
            "single_thread": {"value": 1.0 / t_one, "unit": UNIT, "cores": 1,
                              "sample": f"one evaluation with numpy's FFT on one thread: {t_one:.2f} s"}}


def run_reference(args):
    world, rank, _ = dist_env()
    if rank != 0:
        return 0
    w = wl.WORKLOADS[args.workload]
    n = w["n"]
    cores, model = host_cpu()
    m = wl.vortex(n, w["d"], noise=0.05, seed=1)
    p, setup_s = oracle_setup(w, cores)
    warm = max(1, min(args.warmup, 5))          # warm-up evaluations (each takes seconds)
    t_eval = time_oracle(p, m, warm)
    steps = max(1, min(args.steps, int(args.cpu_budget // max(t_eval, 1e-3))))
    t0 = time.perf_counter()
    for _ in range(steps):
        oracle_field_eval(p, m)
    el = time.perf_counter() - t0
    value = steps / el
    sample = (f"{steps} demag + exchange field evaluations of the {n[0]}x{n[1]}x{n[2]} film (of {args.steps} "
              f"requested, capped to ~{args.cpu_budget:.0f} s of oracle work), float64 numpy with scipy.fft on "
              f"{cores} threads ({model}); {warm} warm-up evaluations; Newell kernel setup ({setup_s:.0f} s) excluded")
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": steps, "warmup": warm, "ms_per_step": 1e3 * el / steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "film512: 512x512x16 cells of 2 nm, permalloy, alpha 0.5, seeded vortex + 5% noise",
                   "what": "CPU oracle field evaluation"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------ GPU arm
DEMAG = ("xfwd", "yfwd", "zconv", "yinv", "xinv")
TIMED = DEMAG + ("stage",)

# float-float cost model: FP32 instructions per operation (mm_ff.cuh: the
# add is TwoSum + low parts + fast two-sum, the multiply TwoProd by FMA +
# two cross FMAs + fast two-sum), and the add/multiply mix of a radix-2 FFT
# butterfly with its complex twiddle (6 adds, 4 multiplies per 10 flops)
FF_ADD_INSTR, FF_MUL_INSTR = 11, 7
# steps of the fully instrumented window before the timed region
PROFILE_STEPS = 20
FF_INSTR_PER_FLOP = (6 * FF_ADD_INSTR + 4 * FF_MUL_INSTR) / 10.0


class Run:
    """One timed stretch of relax() (or the minimiser) on one context."""

    def __init__(self, mm, ctx, m, solver):
        self.mm, self.ctx, self.m, self.solver = mm, ctx, m, solver

    def advance(self, steps):
        mm = self.mm
        try:
            if self.solver == "bb":
                mm.mm_minimize_bb(self.ctx, self.m, torque_tol=0.0, max_iter=steps)
            else:
                mm.mm_relax(self.ctx, self.m, t_max=5e-9, torque_tol=0.0, max_steps=steps)
        except mm.MMError as e:          # stopping on the step cap is the expected outcome here
            if e.code != mm.MM_ERR_NOT_CONVERGED:
                raise

    def timed(self, steps, stream, barrier=None, clocks=None, classes=None):
        """Time `steps` steps with CUDA events on the library's stream.  The
        kernel classes named in `classes` (default: all) get an event pair
        per launch; every class's launches are counted."""
        import torch
        mm = self.mm
        if classes is None:
            mm.mm_enable_kernel_timing(self.ctx, True)
        else:
            mm.mm_enable_kernel_timing_mask(self.ctx, sum(1 << mm.KERNEL_NAMES.index(k) for k in classes))
        launches0 = mm.mm_kernel_launches(self.ctx)
        if barrier:
            barrier()
        torch.cuda.synchronize()
        if clocks:
            clocks.start()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        self.advance(steps)
        ev1.record(stream)
        torch.cuda.synchronize()
        if barrier:
            barrier()
        clk = clocks.stop() if clocks else None
        ms = ev0.elapsed_time(ev1)
        launches = mm.mm_kernel_launches(self.ctx) - launches0
        accepted, rejected, t_sim, _ = mm.mm_step_stats(self.ctx)
        if self.solver == "bb":
            accepted, rejected = steps, 0
        kt = {name: mm.mm_kernel_time(self.ctx, k) for k, name in enumerate(mm.KERNEL_NAMES)}
        mm.mm_enable_kernel_timing(self.ctx, False)
        return {"ms": ms, "evals": kt["zconv"][1], "accepted": accepted, "rejected": rejected, "kt": kt,
                "launches": launches, "clocks": clk}


def kernel_table(kt, n, s):
    out = {}
    for k in TIMED:
        t_ms, cnt = kt[k]
        if cnt:
            b = algorithmic_bytes(k, n, s)
            out[k] = {"launches": cnt, "avg_us": round(1e3 * t_ms / cnt, 2), "algo_MB": round(b / 1e6, 2),
                      "GB_s": round(b / (t_ms / 1e3 / cnt) / 1e9, 1)}
    return out


def path_roofline(kt, n, s, peak):
    """Whole-path HBM view: the algorithmic bytes of every timed demag and
    stage launch over their summed device time."""
    byts = sum(algorithmic_bytes(k, n, s) * kt[k][1] for k in TIMED)
    sec = sum(kt[k][0] for k in TIMED) / 1e3
    if sec <= 0:
        return None
    gbs = byts / sec / 1e9
    return {"kernels": list(TIMED), "algorithmic_GB": byts / 1e9, "kernel_s": sec, "achieved": gbs, "peak": peak,
            "unit": "GB/s", "frac": gbs / peak}


def hbm_roofline(dom, kt, n, s, peak, peak_src, precision):
    tot_ms, nl = kt[dom]
    avg_s = tot_ms / 1e3 / max(nl, 1)
    algo = algorithmic_bytes(dom, n, s)
    achieved = algo / avg_s / 1e9
    return {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": peak, "unit": "GB/s",
            "frac": achieved / peak, "traffic": ncu_traffic(dom, precision), "peak_source": f"{peak_src} (hbm_gbs)",
            "algorithmic_bytes_per_launch": algo}


def alu_roofline(dom, kt, n, peak_tflops, peak_src, hbm):
    tot_ms, nl = kt[dom]
    avg_s = tot_ms / 1e3 / max(nl, 1)
    fl = algorithmic_flops(dom, n)
    tf = fl / avg_s / 1e12
    return {"bound": "alu", "kernel": dom, "achieved": tf, "peak": peak_tflops, "unit": "TFLOP/s",
            "frac": tf / peak_tflops, "traffic": None, "peak_source": peak_src, "algorithmic_flops_per_launch": fl,
            "hbm": hbm}


def measure_f64(mm, w, stream, steps, warmup, peak, peak_src, alu, e2e_steps, cufft_reps=0):
    """The FP64 half of the metric on the same film: float-float passes and
    stage (MM_FFT_FF, the fast FP64 path) and native FP64, each with its
    kernel table and ALU roofline against the measured FMA roofs."""
    import torch
    n, d = w["n"], w["d"]
    N = n[0] * n[1] * n[2]
    m_host = wl.vortex(n, d, noise=0.05, seed=1)
    out = {}
    ctx = mm.mm_init_mesh(*n, *d, precision=mm.MM_F64, stream=stream)
    mm.mm_set_material(ctx, w["Ms"], w["A"], w["alpha"], w["Ku"])
    for name, mode, k_steps, k_warm in (("ff", mm.MM_FFT_FF, steps, warmup), ("native", 0, max(2, steps // 4), 2)):
        mm.mm_set_fft_mode(ctx, mode)
        m = torch.tensor(m_host, dtype=torch.float64, device="cuda")
        run = Run(mm, ctx, m, "relax")
        run.advance(k_warm)
        r = run.timed(k_steps, stream)
        kt = r["kt"]
        dom = max(TIMED, key=lambda k: kt[k][0])
        hbm = hbm_roofline(dom, kt, n, 8, peak, peak_src, traffic_key("f64", "ff" if mode else "fp32"))
        if name == "ff":
            fp32 = alu["fp32_fma_tflops"]
            roof = fp32 / 2.0 / FF_INSTR_PER_FLOP
            src = (f"measured FP32 FMA rate {fp32:.1f} TFLOP/s (mm_alu_peak) / 2 = FP32 instructions/s, divided by "
                   f"{FF_INSTR_PER_FLOP:.1f} FP32 instructions per FP64-equivalent flop in float-float "
                   f"(add {FF_ADD_INSTR}, multiply {FF_MUL_INSTR}; 6 adds + 4 multiplies per butterfly)")
        else:
            roof = alu["fp64_fma_tflops"]
            src = "measured FP64 FMA rate (mm_alu_peak, fma.rn.f64, 2 flops per FMA)"
        roofline = alu_roofline(dom, kt, n, roof, src, hbm) if algorithmic_flops(dom, n) else hbm
        entry = {"value": r["evals"] / (r["ms"] / 1e3), "unit": UNIT, "steps": k_steps, "warmup": k_warm,
                 "ms_per_step": r["ms"] / max(r["accepted"], 1),
                 "llg_mcell_steps_per_s": r["accepted"] * N / (r["ms"] / 1e3) / 1e6,
                 "accepted_steps": r["accepted"], "rejected_trials": r["rejected"], "field_evals": r["evals"],
                 "demag_ms_per_eval": sum(kt[k][0] for k in DEMAG) / max(r["evals"], 1),
                 "roofline": roofline, "path_hbm": path_roofline(kt, n, 8, peak),
                 "kernels": kernel_table(kt, n, 8), "gpu_launches": r["launches"],
                 "fft": "float-float passes and stage on the FP32 pipes" if mode else "native FP64"}
        if name == "ff" and e2e_steps > 0:
            entry["e2e"] = e2e_host(mm, ctx, m_host, torch.float64, min(e2e_steps, 3))
        out[name] = entry
    if cufft_reps:
        out["cufft"] = cufft_compare(mm, ctx, m, w["Ms"], n, cufft_reps)
    mm.mm_destroy(ctx)
    del m
    return out


def e2e_host(mm, ctx, m_host, tdtype, steps):
    """End to end through mm_llg_step_host: each RKF45 step copies m from
    pinned host memory to the device and back inside the call."""
    import torch
    import numpy as np
    pinned = torch.from_numpy(m_host.astype(np.float64 if tdtype == torch.float64 else np.float32)).pin_memory()
    # launches are counted for every class; one class carries events
    mm.mm_enable_kernel_timing_mask(ctx, 1 << mm.KERNEL_NAMES.index("zconv"))
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    t_s, dt_s = 0.0, 1e-14
    for _ in range(steps):
        t_s, dt_s, _ = mm.mm_llg_step_host(ctx, pinned, t_s, dt_s, mm.MM_RKF45, 1e-5)
    el = time.perf_counter() - t0
    evals = mm.mm_kernel_time(ctx, mm.KERNEL_NAMES.index("zconv"))[1]
    mm.mm_enable_kernel_timing(ctx, False)
    nbytes = int(pinned.numel() * pinned.element_size())
    return {"value": evals / el, "unit": UNIT, "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes,
            "steps": steps, "api": "mm_llg_step_host (RKF45): m copied host->device and device->host inside each call"}


def cufft_compare(mm, ctx, m, Ms, n, reps):
    """Demag through cuFFT (torch.fft R2C/C2R on the whole padded grid) with
    the library's k-space product between the transforms: zero-padded M,
    rfftn, -N^ M^, irfftn, crop.  Timed with CUDA events; never on the
    library's path."""
    import torch
    nx, ny, nz = n
    P = (2 * nz if nz > 1 else 1, 2 * ny if ny > 1 else 1, 2 * nx if nx > 1 else 1)
    Mp = torch.zeros((3,) + P, dtype=m.dtype, device=m.device)
    H = torch.empty_like(m)
    spec = None

    def once():
        nonlocal spec
        Mp[:, :nz, :ny, :nx] = m * Ms
        spec = torch.fft.rfftn(Mp, dim=(1, 2, 3)).contiguous()
        mm.mm_kspace_product(ctx, spec)
        H.copy_(torch.fft.irfftn(spec, s=P, dim=(1, 2, 3))[:, :nz, :ny, :nx])

    def ffts_only():
        s_ = torch.fft.rfftn(Mp, dim=(1, 2, 3))
        torch.fft.irfftn(s_, s=P, dim=(1, 2, 3))

    for _ in range(3):
        once()
    torch.cuda.synchronize()
    res = {}
    for name, fn in (("per_eval", once), ("ffts_only", ffts_only)):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        torch.cuda.synchronize()
        res[name] = a.elapsed_time(b) / reps
    # cuFFT's compulsory traffic with unpruned transforms: read the padded M,
    # write its spectrum, read + write it in the product (kernel octant
    # aside), read it for the inverse, write the padded field
    s = m.element_size()
    padded = 3 * P[0] * P[1] * P[2] * s
    spec_b = 3 * P[0] * P[1] * (P[2] // 2 + 1) * 2 * s
    min_bytes = padded + spec_b + 2 * spec_b + spec_b + padded
    out = {"demag_ms_per_eval": res["per_eval"], "ffts_only_ms": res["ffts_only"], "reps": reps,
           "unpruned_min_GB": min_bytes / 1e9, "GB_s_on_unpruned_min": min_bytes / (res["per_eval"] / 1e3) / 1e9,
           "what": "torch.fft rfftn/irfftn (cuFFT) on the padded grid + mm_kspace_product, pad and crop included"}
    del Mp, spec
    torch.cuda.empty_cache()
    return out


def windows(run, steps, count, stream, kernel_timing=True, classes=("zconv",)):
    """Field evals/s of `count` further relax() windows of `steps` steps:
    median and 10th / 90th percentiles, timed like the headline (events
    around the launches of `classes` only).  Without kernel timing the only
    events are those around the step controller's two launches per trial
    (the evaluations are counted from the z-pass launches either way)."""
    import numpy as np
    vals = []
    for _ in range(count):
        r = run.timed(steps, stream, classes=classes if kernel_timing else ("control",))
        vals.append(r["evals"] / (r["ms"] / 1e3))
    return {"windows": count, "steps_each": steps, "median": float(np.median(vals)),
            "p10": float(np.percentile(vals, 10)), "p90": float(np.percentile(vals, 90)),
            "values": [round(v, 1) for v in vals],
            "kernel_timing": ("events around " + ", ".join(classes) + " launches") if kernel_timing
            else "events around the step controller's launches only"}


def measure_alu():
    import paper_2606_01114_gb300 as mm
    return {"fp64_fma_tflops": mm.mm_alu_peak(mm.MM_ROOF_FP64) / 1e12,
            "fp32_fma_tflops": mm.mm_alu_peak(mm.MM_ROOF_FP32) / 1e12,
            "fp32x2_fma_tflops": mm.mm_alu_peak(mm.MM_ROOF_FP32X2) / 1e12,
            "how": "mm_alu_peak: 8 independent FMA chains per thread, 8 blocks per SM, best of 3 launches"}


def run_relax_to(args, mm, ctx, m, n, s, stream, local):
    """One relax() call from the vortex to t_max (adaptive RKF45, tol 1e-5,
    first dt 1e-14 s): wall time, accepted and rejected steps, field
    evaluations, clocks."""
    import torch
    N = n[0] * n[1] * n[2]
    clocks = ClockSampler(local)
    mm.mm_enable_kernel_timing(ctx, True)
    torch.cuda.synchronize()
    clocks.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    t_sim, steps = mm.mm_relax(ctx, m, t_max=args.relax_to, torque_tol=0.0, max_steps=10 ** 8)
    ev1.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    ms = ev0.elapsed_time(ev1)
    accepted, rejected, t_end, dt_last = mm.mm_step_stats(ctx)
    kt = {name: mm.mm_kernel_time(ctx, k) for k, name in enumerate(mm.KERNEL_NAMES)}
    mm.mm_enable_kernel_timing(ctx, False)
    evals = kt["zconv"][1]
    E = mm.mm_energy(ctx, m)
    return {"metric": METRIC, "value": evals / (ms / 1e3), "unit": UNIT, "n_gpus": 1, "higher_is_better": True,
            "dtype": args.precision + ("/ff" if args.fft_mode == "ff" else ""), "data": "synthetic",
            "config": {"workload": f"film512 relaxation to t = {args.relax_to:g} s in one relax() call",
                       "fft": args.fft_mode},
            "relax": {"t_sim": t_end, "accepted_steps": accepted, "rejected_trials": rejected, "field_evals": evals,
                      "wall_s": ms / 1e3, "mean_dt": t_end / max(accepted, 1), "last_dt": dt_last,
                      "llg_mcell_steps_per_s": accepted * N / (ms / 1e3) / 1e6,
                      "energies_J": [float(e) for e in E]},
            "kernels": kernel_table(kt, n, s), "path_hbm": path_roofline(kt, n, s, load_peaks()[0]),
            "clocks": clk}


def run_per_field(args, mm, ctx, m, n, s, stream):
    """The paper's per-field protocol: each field evaluated alone, 1000
    warm-up calls, then `iters` calls each bracketed by CUDA events on the
    library's stream; median, 10th and 90th percentile per call."""
    import numpy as np
    import torch
    H = torch.empty_like(m)
    peak, peak_src = load_peaks()
    demag_bytes = sum(algorithmic_bytes(k, n, s) for k in DEMAG)
    out = {}
    for name, fn in (("demag", mm.mm_demag_field), ("exchange", mm.mm_exchange_field)):
        for _ in range(1000):
            fn(ctx, m, H)
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(args.per_field)]
        torch.cuda.synchronize()
        for a, b in evs:
            a.record(stream)
            fn(ctx, m, H)
            b.record(stream)
        torch.cuda.synchronize()
        us = np.array([a.elapsed_time(b) * 1e3 for a, b in evs])
        e = {"iters": args.per_field, "warmup": 1000, "median_us": float(np.median(us)),
             "p10_us": float(np.percentile(us, 10)), "p90_us": float(np.percentile(us, 90))}
        if name == "demag":
            e["hbm_frac_of_measured_median"] = demag_bytes / (e["median_us"] / 1e6) / 1e9 / peak
            e["algorithmic_GB"] = demag_bytes / 1e9
        out[name] = e
    return {"metric": "per-field time (the paper's benchmark protocol)", "unit": "us per call",
            "dtype": args.precision + ("/ff" if args.fft_mode == "ff" else ""), "data": "synthetic",
            "config": {"workload": "film512: 512x512x16 cells of 2 nm, seeded vortex + 5% noise",
                       "fft": args.fft_mode, "peak_GB_s": peak, "peak_source": peak_src},
            "fields": out}


def run_ours(args):
    import torch
    import paper_2606_01114_gb300 as mm
    from paper_2606_01114_gb300 import build as _build

    world, rank, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group(backend="nccl" if torch.cuda.is_available() else "gloo")
    else:
        dist = None
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA GPU (no CPU fallback)")
    torch.cuda.set_device(local)
    _build.build()
    w = wl.WORKLOADS[args.workload]
    n, d = w["n"], w["d"]
    N = n[0] * n[1] * n[2]
    prec = mm.MM_F64 if args.precision == "f64" else mm.MM_F32
    tdtype = torch.float64 if prec == mm.MM_F64 else torch.float32
    s = 8 if prec == mm.MM_F64 else 4
    stream = torch.cuda.current_stream()
    ctx = mm.mm_init_mesh(*n, *d, precision=prec, stream=stream)
    mm.mm_set_material(ctx, w["Ms"], w["A"], w["alpha"], w["Ku"])
    if args.fft_mode == "ff":
        if prec != mm.MM_F64:
            raise SystemExit("--fft-mode ff needs --precision f64")
        mm.mm_set_fft_mode(ctx, mm.MM_FFT_FF)
    elif args.fft_mode == "f4":
        mm.mm_set_fft_mode(ctx, mm.MM_FFT_F4)
    elif args.fft_mode != "fp32":
        mm.mm_set_fft_mode(ctx, mm.MM_TC_TF32 if args.fft_mode == "tf32" else mm.MM_TC_BF16)
    if args.dmi:
        mm.mm_set_dmi(ctx, args.dmi, mm.MM_DMI_INTERFACIAL)
    if args.stt:
        mm.mm_set_stt(ctx, args.stt, 0.4, 2.0, 0.0, (0.0, 0.0, 1.0))
    m_host = wl.vortex(n, d, noise=0.05, seed=1)
    m = torch.tensor(m_host, dtype=tdtype, device="cuda")

    if args.per_field:
        if rank == 0:
            print(json.dumps(run_per_field(args, mm, ctx, m, n, s, stream)), flush=True)
        mm.mm_destroy(ctx)
        return 0

    if args.relax_to:
        if rank == 0:
            print(json.dumps(run_relax_to(args, mm, ctx, m, n, s, stream, local)), flush=True)
        mm.mm_destroy(ctx)
        return 0

    def barrier():
        if dist is not None:
            dist.barrier()

    run = Run(mm, ctx, m, args.solver)
    run.advance(args.warmup)
    torch.cuda.synchronize()
    # every launch timed over a window before the timed region: the kernel
    # table, the whole-path view, and which kernel dominates
    prof = run.timed(PROFILE_STEPS, stream)
    kt = prof["kt"]
    dom = max(TIMED, key=lambda k: kt[k][0])
    # timed region: device-resident input; only the dominant kernel's launches
    # carry CUDA events (its roofline), so the region is nearly uninstrumented
    r = run.timed(args.steps, stream, barrier=barrier, clocks=ClockSampler(local), classes=(dom,))
    ms, evals, accepted, rejected, kt_run = r["ms"], r["evals"], r["accepted"], r["rejected"], r["kt"]
    ms_max, evals_all, acc_all = reduce_over_ranks(dist, ms, evals, accepted, "cuda")
    value = evals_all / (ms_max / 1e3)
    rate = acc_all * N / (ms_max / 1e3) / 1e6

    peak, peak_src = load_peaks()
    roofline = hbm_roofline(dom, kt_run, n, s, peak, peak_src, traffic_key(args.precision, args.fft_mode))
    extras = rank == 0 and world == 1 and not args.no_extras
    alu = measure_alu() if extras or prec == mm.MM_F64 else None
    if prec == mm.MM_F64 and algorithmic_flops(dom, n):
        if args.fft_mode == "ff":
            roof = alu["fp32_fma_tflops"] / 2.0 / FF_INSTR_PER_FLOP
            src = f"measured FP32 FMA rate / 2 / {FF_INSTR_PER_FLOP:.1f} FP32 instructions per float-float flop"
        else:
            roof, src = alu["fp64_fma_tflops"], "measured FP64 FMA rate (mm_alu_peak)"
        roofline = alu_roofline(dom, kt_run, n, roof, src, roofline)
    prof_evals = kt["zconv"][1]
    demag_ms = sum(kt[k][0] for k in DEMAG)
    demag_bytes = sum(algorithmic_bytes(k, n, s) for k in DEMAG)
    kernel_share = {k: round(v[0] / max(sum(x[0] for x in kt.values()), 1e-9), 4) for k, v in kt.items()}

    # end to end through the public API with host buffers
    e2e = None
    if args.e2e_steps > 0:
        if args.solver == "bb":
            pinned = torch.from_numpy(m_host.astype(np.float64 if prec == mm.MM_F64 else np.float32)).pin_memory()
            mm.mm_enable_kernel_timing_mask(ctx, 1 << mm.KERNEL_NAMES.index("zconv"))
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(args.e2e_steps):
                m.copy_(pinned, non_blocking=True)
                run.advance(1)
                pinned.copy_(m)
            torch.cuda.synchronize()
            el = time.perf_counter() - t0
            ev = mm.mm_kernel_time(ctx, mm.KERNEL_NAMES.index("zconv"))[1]
            mm.mm_enable_kernel_timing(ctx, False)
            nb = int(pinned.numel() * pinned.element_size())
            e2e = {"value": ev / el * world, "unit": UNIT, "h2d_bytes_per_step": nb, "d2h_bytes_per_step": nb,
                   "steps": args.e2e_steps, "api": "mm_minimize_bb (one iteration) per step, m copied by torch"}
        else:
            e2e = e2e_host(mm, ctx, m_host, tdtype, args.e2e_steps)
            e2e["value"] *= world

    line = None
    if rank == 0:
        solver_note = ("Barzilai-Borwein minimiser, one field evaluation per iteration (timed steps = iterations)"
                       if args.solver == "bb" else "relax(): adaptive RKF45")
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / max(accepted, 1), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None,
            "dtype": args.precision + ("/ff" if args.fft_mode == "ff" else ""), "data": "synthetic",
            "config": {"workload": "film512: 512x512x16 cells of 2 nm (padded FFT 1024x1024x32), Ms 8e5 A/m, "
                                   "A 1.3e-11 J/m, alpha 0.5, seeded vortex + 5% noise, adaptive RKF45 tol 1e-5 "
                                   "via relax()",
                       "parallelism": "replicas" if world > 1 else "single GPU",
                       "fft": args.fft_mode, "solver": solver_note, "dmi_D": args.dmi, "stt_J": args.stt,
                       "l2": "no flush: one field evaluation moves ~1.9 GB, far above the 129 MB L2"},
            "accepted_steps": accepted, "rejected_trials": rejected, "field_evals": evals,
            "demag_ms_per_eval": demag_ms / max(prof_evals, 1),
            "demag_GB_s": demag_bytes / (demag_ms / 1e3 / max(prof_evals, 1)) / 1e9,
            "roofline": roofline,
            "path_hbm": path_roofline(kt, n, s, peak),
            "step_hbm_frac": (sum(algorithmic_bytes(k, n, s) * kt_run[k][1] for k in TIMED) / 1e9
                              / (ms / 1e3) / peak),
            "kernels": kernel_table(kt, n, s), "kernel_time_share": kernel_share,
            "kernel_timing": {"timed_region": f"CUDA events around every {dom} launch only",
                              "kernels": f"every launch timed over {PROFILE_STEPS} steps before the timed region "
                                         "(kernels, kernel_time_share, path_hbm, demag_ms_per_eval)"},
            "clocks": r["clocks"], "e2e": e2e, "gpu_launches": r["launches"],
        }
        if args.solver == "bb":
            line["mcell_iterations_per_s"] = acc_all * N / (ms_max / 1e3) / 1e6
            line["llg_mcell_steps_per_s"] = None
        else:
            line["llg_mcell_steps_per_s"] = rate
        if alu:
            line["alu_peaks"] = alu

    if extras:
        line["windows"] = windows(run, 20, 5, stream, classes=(dom,))
        if args.solver == "relax":
            line["windows_controller_events_only"] = windows(run, 20, 5, stream, kernel_timing=False)
        if args.solver == "relax" and prec == mm.MM_F32 and args.fft_mode == "fp32" and not (args.dmi or args.stt):
            line["cufft"] = {"f32": cufft_compare(mm, ctx, m, w["Ms"], n, 20)}
            line["cufft"]["f32"]["ours_demag_ms_per_eval"] = line["demag_ms_per_eval"]
            mm.mm_destroy(ctx)
            ctx = None
            del m
            torch.cuda.empty_cache()
            f64 = measure_f64(mm, w, stream, max(5, min(args.steps, 20)), 3, peak, peak_src, alu, args.e2e_steps,
                              cufft_reps=5)
            line["cufft"]["f64"] = f64.pop("cufft")
            line["cufft"]["f64"]["ours_ff_demag_ms_per_eval"] = f64["ff"]["demag_ms_per_eval"]
            line["cufft"]["f64"]["ours_native_demag_ms_per_eval"] = f64["native"]["demag_ms_per_eval"]
            line["f64"] = f64
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w, m_host)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if ctx is not None:
        mm.mm_destroy(ctx)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.ingest_ncu:
        return ingest_ncu(args.ingest_ncu, traffic_key(args.precision, args.fft_mode), "film512 512x512x16 " + args.precision.upper())
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
