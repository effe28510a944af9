"""Benchmark of the FCM pixel pass on GB300.

Workload (one "step" = one whole FCM segmentation, Algorithm 1 of
arXiv:1601.00072, to convergence): the 256^3 uint8 ellipsoid phantom with a
+/-20 % bias field and Rician-like noise (sigma 6), cast to FP32, C = 4,
m = 2, eps = 1e-5 on max|dU|, max_iter = 300, initial U drawn from a seeded
uniform Dirichlet (seed 103). Inputs (x, U^0) are resident in HBM before the
timed region; each step reads U^0 (read only) and writes U^k and V^k.

Metric: pixel-iterations per second (n x iterations, summed over steps and
ranks, over the max-over-ranks timed duration). The working set (x 67 MB,
U^0 268 MB, U 268 MB) exceeds the 129 MB L2, so no flush is needed between
steps.

With ``--gpus N`` under torchrun every rank runs its own copy of the workload
(weak scaling; the pass has no cross-GPU exchange when images are independent).

The line also carries ``batched``: images/s of the 512-slice batch (sides
log-uniform 64..512, C in {3, 4, 5}, m = 2, eps = 1e-5) run cold (seeded
Dirichlet U0, one persistent launch in a CUDA graph) and warm (the shipped
network predicts V^0), each with inputs resident in HBM. A warm slice that
fails the acceptance rule (centers within 1e-4 of the cold start's, or a final
J no larger) is charged its cold start on top: the time it adds to a cold
batch (headline), and, reported beside it, the time of rerunning the failed
slices as a batch of their own. ``batched.histogram_domain`` times the same
cold batch through the histogram-domain path (one CTA per slice).

``--impl reference`` times the FP64 CPU oracle instead, on a bounded sample of
the same workload (rank 0 only).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "volume256"
C = 4
EPS = 1e-5
MAX_ITER = 300
METRIC = "FCM pixel-iterations/s (256^3 volume, C=4, m=2, eps=1e-5)"
UNIT = "pixel-iter/s"
PROFILE = os.path.join(ROOT, "profiles", "fcm_pass_volume256.md")
KERNEL_SOURCES = ["paper_1601_00072_gb300/csrc/fcm_run_inst.cu",
                  "paper_1601_00072_gb300/csrc/fcm_device.cuh",
                  "paper_1601_00072_gb300/csrc/fcm_df.cuh",
                  "paper_1601_00072_gb300/csrc/fcm_run.h",
                  "paper_1601_00072_gb300/csrc/fcm_internal.h"]


def kernel_hash() -> str:
    h = hashlib.sha256()
    for rel in KERNEL_SOURCES:
        with open(os.path.join(ROOT, rel), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def source_hash(files) -> str:
    h = hashlib.sha256()
    for rel in files:
        with open(os.path.join(ROOT, rel), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def profiled_instructions(path, sources):
    """Warp instructions per launch from a committed ncu summary, if it was
    taken on the current kernel sources; else None."""
    try:
        text = open(os.path.join(ROOT, path)).read()
    except OSError:
        return None
    mh = re.search(r"kernel source hash:\s*`?([0-9a-f]{16})", text)
    mt = re.search(r"warp instructions per launch:\s*([0-9]+)", text)
    line = next((ln for ln in text.splitlines() if ln.startswith("One launch")), "")
    mi = re.search(r"([0-9]+) iterations", line)
    if not mh or not mt or mh.group(1) != source_hash(sources):
        return None
    return float(mt.group(1)), (int(mi.group(1)) if mi else None)


def issue_roofline(path, sources, ms, iters, sm_mhz):
    """ALU-issue roofline of a kernel: warp instructions per launch (from its
    committed ncu summary, for the same iteration count) over the live time,
    against SMs x 4 schedulers x the SM clock."""
    import torch
    got = profiled_instructions(path, sources)
    if got is None or got[1] != iters:
        return None
    inst, _ = got
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    peak = sms * 4 * (sm_mhz or 2070.0) * 1e6 / 1e9
    achieved = inst / (ms / 1e3) / 1e9
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "G warp-instr/s", "frac": achieved / peak,
            "instructions_per_launch": inst, "source": path,
            "peak_source": f"{sms} SMs x 4 schedulers x {sm_mhz or 2070.0:.0f} MHz"}


def fp32_ops_per_pixel_iter(C, m):
    """FP32 operations of a sums pass per pixel (packed pairs count as two):
    differences C, squares C (none at m = 3), co-products 3 (C - 2), their sum
    C - 1, u^m 2C (one more C at m = 3 and 1.5), numerators and denominators 2C."""
    ops = C + 3 * max(C - 2, 0) + (C - 1) + 2 * C + 2 * C
    ops += 0 if m == 3.0 else C
    ops += C if m in (1.5, 3.0) else 0
    return ops


def fp32_roofline(px_iters, ms, C, m, sm_mhz):
    """Of the FP32 pipe: 128 lanes per SM and clock."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    mhz = sm_mhz or 2070.0
    peak = sms * 128 * mhz * 1e6 / 1e12
    achieved = px_iters * fp32_ops_per_pixel_iter(C, m) / (ms / 1e3) / 1e12
    return {"bound": "fp32 pipe", "achieved": achieved, "peak": peak, "unit": "T FP32 instr/s", "frac": achieved / peak,
            "ops_per_pixel_iter": fp32_ops_per_pixel_iter(C, m),
            "peak_source": f"{sms} SMs x 128 lanes x {mhz:.0f} MHz"}


def measured_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def profiled_traffic():
    """DRAM bytes per launch of the iteration kernel from the committed ncu
    summary, if it was taken on the current kernel source; else None."""
    try:
        text = open(PROFILE).read()
    except OSError:
        return None
    mh = re.search(r"kernel source hash:\s*`?([0-9a-f]{16})", text)
    mt = re.search(r"dram bytes per launch:\s*([0-9.eE+]+)", text)
    if not mh or not mt or mh.group(1) != kernel_hash():
        return None
    return float(mt.group(1))


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during a region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        self.lines = []
        self.error = None

    def start(self):
        import torch
        ident = str(self.dev)
        try:
            uuid = str(torch.cuda.get_device_properties(self.dev).uuid)
            ident = uuid if uuid.startswith("GPU-") else "GPU-" + uuid
        except Exception:
            pass
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", ident, f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception as e:  # nvidia-smi missing
            self.error = str(e)
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()
        time.sleep(0.3)

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.15)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.lines:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[3:7]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup():
    """Rank, world size and local rank from the launcher's environment; joins
    the process group (NCCL on GPUs, gloo on a machine without them)."""
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
            dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        else:
            dist.init_process_group("gloo")
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def allreduce(value: float, op: str, world: int) -> float:
    if world == 1:
        return value
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([value], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX if op == "max" else dist.ReduceOp.SUM)
    return float(t.item())


def workload_name(m: float) -> str:
    return ("256^3 uint8 ellipsoid phantom (bias +/-20 percent, Rician sigma 6) as f32, "
            f"C=4, m={m:g}, eps=1e-5, max_iter=300, Dirichlet U0 seed 103")


def load_workload(m: float, with_labels: bool = False):
    import phantom
    x, lab, u0, c = phantom.single_image(WORKLOAD)
    assert c == C
    return (x, u0, lab) if with_labels else (x, u0)


def cpu_sample(x, u0):
    """The bounded CPU sample: the 16 middle slices (1,048,576 voxels)."""
    plane = 256 * 256
    lo, hi = 120 * plane, 136 * plane
    return x[lo:hi], np.ascontiguousarray(u0[:, lo:hi]), "voxels of slices z=120..135 (1,048,576 voxels)"


def run_cpu_oracle_sample(x, u0, m: float, iters: int):
    """The FP64 oracle, as it stands, on the sample for a fixed iteration count."""
    import oracle
    xs, us, desc = cpu_sample(x, u0)
    t0 = time.perf_counter()
    r = oracle.fcm(xs.astype(np.float64), C, m, 0.0, iters, U0=us, want_U=False)
    dt = time.perf_counter() - t0
    return xs.size * r["iters"] / dt, f"{desc}, {r['iters']} iterations (eps=0)", dt


def _oracle_worker_ready(_):
    import oracle
    oracle.lib()
    return os.getpid()


def _oracle_slab(job):
    """One worker of the all-cores timing: the single-thread oracle, as it
    stands, on its own slab; the clock runs inside the worker."""
    xs, us, m, iters = job
    import oracle
    t0 = time.perf_counter()
    r = oracle.fcm(xs, C, m, 0.0, iters, U0=us, want_U=False)
    return xs.size * r["iters"], time.perf_counter() - t0


def run_cpu_oracle_all_cores(x, u0, m: float, iters: int = 30):
    """The oracle on every host core at once: one independent single-thread
    run per core, each on its own 4-slice slab of the volume (262,144 voxels,
    a fixed iteration count), in spawned processes. Throughput = all the
    workers' pixel-iterations over the wall time of the concurrent runs."""
    import multiprocessing as mp
    cores = len(os.sched_getaffinity(0))
    plane = 256 * 256
    jobs = []
    for w in range(cores):
        z0 = 8 + (15 * w) % 240
        lo, hi = z0 * plane, (z0 + 4) * plane
        jobs.append((x[lo:hi].astype(np.float64), np.ascontiguousarray(u0[:, lo:hi]), m, iters))
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(_oracle_worker_ready, range(cores), chunksize=1)
        t0 = time.perf_counter()
        res = pool.map(_oracle_slab, jobs, chunksize=1)
        wall = time.perf_counter() - t0
    units = sum(r[0] for r in res)
    return {"value": units / wall, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{cores} concurrent single-thread runs, each 262,144 voxels (4 slices) x {iters} "
                      "iterations (eps=0); wall time includes handing each worker its slab",
            "seconds": round(wall, 2), "worker_seconds_max": round(max(r[1] for r in res), 2)}


def _center_err(v, ref):
    v, ref = np.asarray(v, np.float64).reshape(-1), np.asarray(ref, np.float64).reshape(-1)
    return float(np.max(np.abs(v - ref) / np.maximum(np.abs(ref), 1.0)))


def _exact_U_vs_bins(Udev, x_u8, Vref, m):
    """max|dU| and argmax-label agreement over EVERY pixel: the reference U is
    the oracle's Eq. 4 at the 256 grey levels (a pixel's memberships depend on
    its grey level only), the CUDA U is read back in chunks."""
    import oracle
    Ub = oracle.memberships(np.arange(256.0), np.asarray(Vref, np.float64), m)
    lab_b = np.argmax(Ub, 0)
    n = x_u8.size
    dmax, agree = 0.0, 0
    for lo in range(0, n, 1 << 22):
        hi = min(n, lo + (1 << 22))
        g = Udev[:, lo:hi].cpu().numpy().astype(np.float64)
        xx = x_u8[lo:hi]
        dmax = max(dmax, float(np.max(np.abs(g - Ub[:, xx]))))
        agree += int(np.sum(np.argmax(g, 0) == lab_b[xx]))
    return dmax, agree / n


def _single_precision(x_u8, u0, m, g_iters, g_V, g_J, Udev, what):
    """A single-image result against the FP64 oracle (256-bin form, exact for
    8-bit data) at the CUDA run's own iteration count."""
    import oracle
    eps = float(np.float32(EPS))
    o = oracle.fcm_quantized(x_u8, C, m, eps, MAX_ITER, U0=u0, want_U=False)
    at = o if o["iters"] == g_iters else oracle.fcm_quantized(x_u8, C, m, 0.0, g_iters, U0=u0, want_U=False)
    dU, agree = _exact_U_vs_bins(Udev, x_u8, at["V"], m)
    return {"vs": f"FP64 oracle (256-bin form), same x and U0, at the {what}'s iteration count",
            "center_rel_err": _center_err(g_V, at["V"]), "max_abs_dU": dU, "dU_over": "every pixel",
            "label_agreement": agree, "d_iters": int(g_iters - o["iters"]),
            "J_rel_err": float(abs(g_J - at["J"][-1]) / abs(at["J"][-1]))}


def _batch_precision(slices, host, Cs, refs):
    """Per-slice errors of a batch against the oracle's 256-bin runs at each
    slice's own iteration count: worst and median center error, worst max|dU|
    over every pixel, worst label agreement, the spread of the iteration
    counts. ``refs[i]`` is (U0, V0) of the oracle start of slice i."""
    import oracle
    eps = float(np.float32(EPS))
    ce, du, la, di = [], [], [], []
    for s, (x, _), Cj, (u0, v0) in zip(slices, host, Cs, refs):
        o = oracle.fcm_quantized(x, Cj, 2.0, eps, MAX_ITER, U0=u0, V0=v0, want_U=False)
        at = o if o["iters"] == s.iters else oracle.fcm_quantized(x, Cj, 2.0, 0.0, s.iters, U0=u0, V0=v0,
                                                                    want_U=False)
        Ub = oracle.memberships(np.arange(256.0), at["V"], 2.0)
        g = s.U.cpu().numpy().astype(np.float64)
        ce.append(_center_err(s.V64[:Cj], at["V"]))
        du.append(float(np.max(np.abs(g - Ub[:, x]))))
        la.append(float(np.mean(np.argmax(g, 0) == np.argmax(Ub, 0)[x])))
        di.append(int(s.iters - o["iters"]))
    ce, du, la, di = map(np.asarray, (ce, du, la, di))
    strict = (ce <= 1e-5) & (du <= 1e-5) & (la >= 0.9999) & (np.abs(di) <= 1)
    out = {"center_rel_err": {"max": float(ce.max()), "median": float(np.median(ce))},
           "max_abs_dU": {"max": float(du.max()), "median": float(np.median(du)), "over": "every pixel"},
           "label_agreement_min": float(la.min()), "d_iters": {"min": int(di.min()), "max": int(di.max())},
           "slices_within_all_bars": int(strict.sum()), "slices": int(strict.size),
           "slices_outside": [int(i) for i in np.flatnonzero(~strict)]}
    # a slice outside the bars at the same iterate: its FP32 trajectory left
    # the oracle's (these slices are trajectory-sensitive: the FP64 oracle
    # itself, restarted from its V^1 perturbed at the FP32 rounding scale,
    # converges elsewhere or relabels). Compared on converged results, with
    # clusters matched by sorted centers, against the oracle restarted from
    # V^1 perturbed by +-1e-6 (the spread the tests allow for)
    conv = {}
    for i in np.flatnonzero(~strict):
        s, (x, _), Cj, (u0, v0) = slices[i], host[i], Cs[i], refs[i]
        o = oracle.fcm_quantized(x, Cj, 2.0, eps, MAX_ITER, U0=u0, V0=v0, want_U=False)
        Ub = oracle.memberships(np.arange(256.0), o["V"], 2.0)
        g = s.U.cpu().numpy().astype(np.float64)
        pg, po = np.argsort(np.asarray(s.V64[:Cj])), np.argsort(o["V"])
        conv[int(i)] = {"center_rel_err_sorted": _center_err(np.asarray(s.V64[:Cj])[pg], o["V"][po]),
                        "max_abs_dU_sorted": float(np.max(np.abs(g[pg] - Ub[po][:, x]))),
                        "J_rel_diff": float((s.J - o["J"][-1]) / abs(o["J"][-1])),
                        "iters": int(s.iters), "oracle_iters": int(o["iters"])}
    if conv:
        out["outside_on_converged_results"] = conv
    return out


def cpu_baseline_leg(x, u0, m, keep, out):
    """Everything that touches the oracle: its timed CPU throughput on a
    bounded sample, and the FP64 reference of every GPU result of the line
    for its precision block (written into ``out``)."""
    import oracle
    value, sample, dt = run_cpu_oracle_sample(x, u0, m, iters=30)
    base = {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": sample, "seconds": round(dt, 2),
            "all_cores": run_cpu_oracle_all_cores(x, u0, m)}
    Ud, Vd, g_iters, g_J = keep["main"]
    out["precision"] = _single_precision(x, u0, m, g_iters, Vd.cpu().numpy(), g_J, Ud, "CUDA run")
    for key, ent in out.get("other_workloads", {}).items():
        Uw, Vw, it, J, xw, u0w, mm = keep[key]
        if key == "phantom200":  # small enough for the per-pixel form of the oracle
            eps = float(np.float32(EPS))
            o = oracle.fcm(xw.astype(np.float64), C, mm, eps, MAX_ITER, U0=u0w, want_U=False)
            at = o if o["iters"] == it else oracle.fcm(xw.astype(np.float64), C, mm, 0.0, it, U0=u0w)
            if "U" not in at or at["U"] is None:
                at = oracle.fcm(xw.astype(np.float64), C, mm, 0.0, it, U0=u0w)
            g = Uw.cpu().numpy().astype(np.float64)
            ent["precision"] = {"vs": "FP64 oracle (per-pixel form), same x and U0, at the CUDA run's iteration count",
                                "center_rel_err": _center_err(Vw.cpu().numpy(), at["V"]),
                                "max_abs_dU": float(np.max(np.abs(g - at["U"]))), "dU_over": "every pixel",
                                "label_agreement": float(np.mean(np.argmax(g, 0) == np.argmax(at["U"], 0))),
                                "d_iters": int(it - o["iters"]),
                                "J_rel_err": float(abs(J - at["J"][-1]) / abs(at["J"][-1]))}
        else:
            ent["precision"] = _single_precision(xw, u0w, mm, it, Vw.cpu().numpy(), J, Uw, "CUDA run")
    if out.get("histogram_domain") and "histogram_domain" in keep:
        Uh, Vh, it, J = keep["histogram_domain"]
        out["histogram_domain"]["precision"] = _single_precision(x, u0, m, it, Vh.cpu().numpy(), J, Uh,
                                                                 "histogram run")
    if out.get("recompute") and "recompute" in keep:
        Ur, Vr, it, J = keep["recompute"]
        out["recompute"]["precision"] = _single_precision(x, u0, m, it, Vr.cpu().numpy(), J, Ur, "U-free run")
    if out.get("multi_feature") and "multi_feature" in keep:
        xm, u0m, Um, rm = keep["multi_feature"]
        eps = float(np.float32(EPS))
        xm64 = xm.astype(np.float64)
        o = oracle.fcm_multi(xm64, C, m, eps, MAX_ITER, U0=u0m)
        at = o if o["iters"] == rm.iters else oracle.fcm_multi(xm64, C, m, 0.0, rm.iters, U0=u0m)
        g = Um.cpu().numpy().astype(np.float64)
        out["multi_feature"]["precision"] = {
            "vs": "FP64 multi-feature oracle, same x and U0, at the CUDA run's iteration count",
            "center_rel_err": _center_err(np.asarray(rm.V64), at["V"]),
            "max_abs_dU": float(np.max(np.abs(g - at["U"]))), "dU_over": "every pixel",
            "label_agreement": float(np.mean(np.argmax(g, 0) == np.argmax(at["U"], 0))),
            "d_iters": int(rm.iters - o["iters"])}
    if out.get("batched") and "batched" in keep:
        cold, warm, hist, host, Cs, cold_p = keep["batched"]
        cold_refs = [(u, None) for _, u in host]
        out["batched"]["cold"]["precision"] = _batch_precision(cold, host, Cs, cold_refs)
        out["batched"]["cold_presolved"]["precision"] = _batch_precision(cold_p, host, Cs, cold_refs)
        out["batched"]["histogram_domain"]["precision"] = _batch_precision(hist, host, Cs, cold_refs)
        # warm slices against the oracle started from the oracle's own
        # prediction (the shipped network in FP64 with its BF16 weights);
        # slices that ran cold against the cold oracle
        from oracle import mlp
        from paper_1601_00072_gb300 import warmstart
        raw = open(warmstart.MODEL_PATH, "rb").read()
        P = mlp.unflat(np.frombuffer(raw[20:], dtype=np.float32).astype(np.float64))
        for k in ("W1", "W2", "W3"):
            b = np.ascontiguousarray(P[k], dtype=np.float32).view(np.uint32).astype(np.uint64)
            P[k] = ((b + 0x7FFF + ((b >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32).astype(np.float64)
        X = np.stack([mlp.features(xh, Cj) for (xh, _), Cj in zip(host, Cs)])
        V0 = mlp.predict_centers(P, X, Cs)
        warm_refs = [((None, np.asarray(v0, np.float32).astype(np.float64)) if s.init == "V" else (u, None))
                     for s, (_, u), v0 in zip(warm, host, V0)]
        out["batched"]["warm"]["precision"] = _batch_precision(warm, host, Cs, warm_refs)
        out["batched"]["warm"]["precision"]["vs"] = (
            "warm slices: FP64 oracle from the oracle's own V0 (the shipped network in FP64 with BF16 weights); "
            "slices that ran cold: FP64 oracle from U0; each at the slice's own iteration count")
    return base


def batch_inputs(dev, n=512, host=None):
    """Device-resident x and U0 of the batch slices (generated in spawned
    worker processes); ``host`` (a list) receives the (x uint8, U0) pairs."""
    import torch
    from paper_1601_00072_gb300 import warmstart
    xs, u0s, Cs = [], [], []
    for part in warmstart.slices_of(range(n), 1):
        for _, Cj, x, u0 in part:
            xs.append(torch.from_numpy(x.astype(np.float32)).to(dev))
            u0s.append(torch.from_numpy(u0[0]).to(dev))
            Cs.append(Cj)
            if host is not None:
                host.append((x, u0[0]))
    return xs, u0s, Cs


def bench_batched(h, dev, steps, warmup, plan=None, keep_results=False, n_slices=512):
    """Cold versus warm-started batch, timed with CUDA events on the launching
    stream (each call returns after its results are read back). ``plan``
    (a dict of FCM.set_batched_plan arguments) replaces the autotuner. With
    ``keep_results`` also returns the slices (results on the device) and the
    host inputs, for the precision report."""
    import torch
    from paper_1601_00072_gb300 import warmstart
    from paper_1601_00072_gb300.fcm import Batch, Slice
    host = []
    xs, u0s, Cs = batch_inputs(dev, n=n_slices, host=host)
    n_img = len(xs)
    px = sum(int(x.numel()) for x in xs)
    cold = [Slice(x=x, C=c, U0=u) for x, c, u in zip(xs, Cs, u0s)]
    h.model_load(warmstart.MODEL_PATH)
    stream = torch.cuda.current_stream(dev)

    spread = {}  # median and largest of the single calls behind each mean

    def timed(fn, reps, name):
        for _ in range(warmup):
            fn()
        torch.cuda.synchronize(dev)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(reps + 1)]
        ev[0].record(stream)
        for e in ev[1:]:
            fn()
            e.record(stream)
        torch.cuda.synchronize(dev)
        each = [a.elapsed_time(b) for a, b in zip(ev, ev[1:])]
        spread[name] = {"ms_median": float(np.median(each)), "ms_max": float(max(each))}
        return ev[0].elapsed_time(ev[-1]) / reps

    if plan:
        h.set_batched_plan(**plan)
    cold = Batch(cold)
    # results land in each Batch's host array; the Slice fields are filled
    # once after timing (the warm call's judge and reruns are inside its time)
    ms_cold = timed(lambda: h.run_batched(cold, read_back=False), steps, "cold")
    cold.read_back()
    plan_used = h.batched_plan()
    # the same cold batch, ordered and split by cost: each slice's iteration
    # count comes from a run on its grey-level histogram inside the call
    cold_p = Batch([Slice(x=x, C=c, U0=u) for x, c, u in zip(xs, Cs, u0s)])
    ms_cold_p = timed(lambda: h.run_batched(cold_p, read_back=False, presolve=True), steps, "cold_presolved")
    cold_p.read_back()
    plan_cold_p = h.batched_plan()
    warm = Batch([Slice(x=x, C=c, U0=u) for x, c, u in zip(xs, Cs, u0s)])
    n_ran_cold = [0]

    def run_warm():
        n_ran_cold[0] = h.run_batched_warm(warm, read_back=False)[1]

    ms_warm = timed(run_warm, steps, "warm")
    warm.read_back()
    plan_warm = h.batched_plan()
    # every returned slice against the cold batch by the acceptance rule; the
    # judge inside the call already ran cold (and timed) each slice whose warm
    # fixed point fails it, so a failure here is a slice whose FP32 per-pixel
    # trajectory left the fixed point the histogram judge saw: it is charged
    # a separate cold batch of its own
    ok = warmstart.accepted(cold.slices, warm.slices)
    bad_i = np.flatnonzero(~ok)
    ms_charge = 0.0
    if bad_i.size:
        bad = Batch([Slice(x=xs[i], C=Cs[i], U0=u0s[i]) for i in bad_i])
        ms_charge = timed(lambda: h.run_batched(bad, read_back=False), steps, "charged")
    it_c = np.array([s.iters for s in cold.slices])
    it_w = np.array([s.iters for s in warm.slices])
    ran_cold = np.array([s.init == "U" for s in warm.slices])
    cold_ips = n_img / (ms_cold / 1e3)
    warm_ips = n_img / ((ms_warm + ms_charge) / 1e3)
    # the same cold batch on each slice's 256-bin histogram (one CTA per
    # slice): the same iterates up to rounding, compared with the cold run
    hist = Batch([Slice(x=x, C=c, U0=u) for x, c, u in zip(xs, Cs, u0s)])
    ms_hist = timed(lambda: h.run_batched_hist(hist, read_back=False), steps, "histogram_domain")
    hist.read_back()
    it_h = np.array([s.iters for s in hist.slices])
    verr = np.array([np.max(np.abs(np.asarray(a.V64) - np.asarray(c.V64)) / np.maximum(np.abs(np.asarray(c.V64)), 1.0))
                     for a, c in zip(hist.slices, cold.slices)])
    res = {
        "workload": f"{n_img} phantom slices, sides log-uniform 64..512, C in {{3,4,5}}, m=2, eps=1e-5, max_iter=300",
        "pixels": px, "steps": steps,
        "cold": {"images_per_s": cold_ips, "ms": ms_cold, "mean_iters": float(it_c.mean()),
                 "max_iters": int(it_c.max()),
                 "pixel_iter_per_s": sum(int(x.numel()) * int(i) for x, i in zip(xs, it_c)) / (ms_cold / 1e3)},
        "warm": {"images_per_s": warm_ips, "ms": ms_warm, "charged_ms": ms_charge,
                 "call": "fcm_run_batched_warm: prediction, histogram-domain judge of every slice (from U0 "
                         "and from the predicted V0), the batch ordered by the judge's iteration counts, "
                         "and cold reruns of rejected warm results, all inside the timed call",
                 "mean_iters": float(it_w.mean()), "max_iters": int(it_w.max()),
                 "mean_iters_of_warm_slices": float(it_w[~ran_cold].mean()) if (~ran_cold).any() else None,
                 "accepted": float(ok.mean()), "failed_slices": int(bad_i.size),
                 "ran_cold_at_run_time": int(n_ran_cold[0])},
        "cold_presolved": {"images_per_s": n_img / (ms_cold_p / 1e3), "ms": ms_cold_p,
                           "call": "fcm_run_batched with FCM_BATCH_PRESOLVE: every slice first runs to convergence "
                                   "on its grey-level histogram from its U0, inside the timed call, and the pixel "
                                   "batch is ordered and split by the iterations that took",
                           "mean_iters": float(np.mean([s.iters for s in cold_p.slices])), "plan": plan_cold_p},
        "warm_over_cold": warm_ips / cold_ips,
        "warm_over_cold_presolved": warm_ips / (n_img / (ms_cold_p / 1e3)),
        "warm_over_cold_presolved_medians": spread["cold_presolved"]["ms_median"] / (spread["warm"]["ms_median"] + ms_charge),
        "plan": plan_used,
        "plan_warm": plan_warm,
        "histogram_domain": {
            "kernel": "k_bins_*: pixel passes in 8,192-pixel chunks over the whole GPU (histogram and V^1 "
                      "sums; the first stop over every pixel only where a bound cannot decide it; U by lookup), "
                      "the iterations on 256 bins, one CTA per slice",
            "images_per_s": n_img / (ms_hist / 1e3), "ms": ms_hist, "speedup_vs_cold": ms_cold / ms_hist,
            "mean_iters": float(it_h.mean()), "max_iters": int(it_h.max()),
            "iters_within_1_of_cold": float(np.mean(np.abs(it_h - it_c) <= 1)),
            "center_rel_err_vs_cold": {"max": float(verr.max()), "fraction_within_1e-5": float(np.mean(verr <= 1e-5))}},
    }
    for name, v in spread.items():
        if name in res:
            res[name].update(v)
    if keep_results:
        return res, (cold.slices, warm.slices, hist.slices, host, Cs, cold_p.slices)
    return res


def bench_ours(args):
    import torch

    world, rank, local = dist_setup()
    torch.cuda.set_device(local)
    from paper_1601_00072_gb300 import _build
    if rank == 0 or world == 1:
        _build.build()
    barrier(world)
    from paper_1601_00072_gb300.fcm import FCM

    m = args.m
    x, u0, lab = load_workload(m, with_labels=True)
    n = x.size
    dev = torch.device("cuda", local)
    xd = torch.from_numpy(x.astype(np.float32)).to(dev)
    U0d = torch.from_numpy(u0).to(dev)
    Ud = torch.empty_like(U0d)
    Vd = torch.empty(C, dtype=torch.float32, device=dev)
    h = FCM(local)
    stream = torch.cuda.current_stream(dev)

    def step():
        return h.run(xd, C, m, EPS, MAX_ITER, U0=U0d, U=Ud, V=Vd, graph=not args.no_graph,
                     tma=args.variant == "tma")

    for _ in range(args.warmup):
        r = step()
    torch.cuda.synchronize(dev)

    sampler = ClockSampler(local)
    sampler.start()
    barrier(world)
    torch.cuda.synchronize(dev)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    # one event per step boundary as well, for the per-run mean/median/min the
    # paper's protocol reports (the events add no work to the stream)
    marks = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    e0.record(stream)
    marks[0].record(stream)
    iters = []
    launches = 0
    for k in range(args.steps):
        r = step()
        marks[k + 1].record(stream)
        iters.append(r.iters)
        launches += r.launches
    e1.record(stream)
    torch.cuda.synchronize(dev)
    barrier(world)
    clocks = sampler.stop()
    ms_local = e0.elapsed_time(e1)
    per_step = [marks[k].elapsed_time(marks[k + 1]) for k in range(args.steps)]
    ms = allreduce(ms_local, "max", world)
    units_local = float(n) * sum(iters)
    units = allreduce(units_local, "sum", world)
    value = units / (ms / 1e3)

    # rooflines over the timed region: the FP32 pipe bounds the iterations, which
    # read x alone (from shared memory and the L2); HBM the first pass (x and U^0)
    # and the last (U^k written once)
    bytes_local = sum((4 * n + 4 * C * n) + (4 * n + 4 * C * n) for _ in iters)
    hbm_gbs = bytes_local / (ms_local / 1e3) / 1e9
    peak, peak_kind = measured_peak()
    traffic = profiled_traffic()

    # end to end through the C ABI with host buffers. Headline: a sequence of
    # steps in one fcm_run_stream call, each step's H2D of x and U^0 and D2H
    # of U^k and V^k overlapped with the neighbouring steps' runs. Beside it:
    # one synchronous fcm_run call per step (copies, run, copies).
    e2e = None
    if not args.no_e2e:
        xh = torch.from_numpy(x.astype(np.float32)).pin_memory()
        U0h = torch.from_numpy(u0).pin_memory()
        Uh = [torch.empty_like(U0h).pin_memory() for _ in range(2)]
        Vh = torch.empty(C, dtype=torch.float32).pin_memory()
        e_steps = max(3, min(args.steps, 20))
        h.run_stream([xh, xh], C, m, EPS, MAX_ITER, U0s=[U0h, U0h], Us=Uh)
        barrier(world)
        t0 = time.perf_counter()
        rs = h.run_stream([xh] * e_steps, C, m, EPS, MAX_ITER, U0s=[U0h] * e_steps,
                          Us=[Uh[k % 2] for k in range(e_steps)])
        dt = time.perf_counter() - t0
        e_units = sum(n * rr.iters for rr in rs)
        dt = allreduce(dt, "max", world)
        e_units = allreduce(float(e_units), "sum", world)
        # one synchronous call per step
        h.run(xh, C, m, EPS, MAX_ITER, U0=U0h, U=Uh[0], V=Vh)
        s_steps = max(3, min(args.steps, 10))
        barrier(world)
        t1 = time.perf_counter()
        s_units = 0
        for _ in range(s_steps):
            rr = h.run(xh, C, m, EPS, MAX_ITER, U0=U0h, U=Uh[0], V=Vh)
            s_units += n * rr.iters
        dt1 = allreduce(time.perf_counter() - t1, "max", world)
        s_units = allreduce(float(s_units), "sum", world)
        e2e = {"value": e_units / dt, "unit": UNIT,
               "h2d_bytes_per_step": 4 * n + 4 * C * n,
               "d2h_bytes_per_step": 4 * C * n + 4 * C,
               "api": f"fcm_run_stream: {e_steps} steps in one call from pinned host memory, the copies "
                      "of each step overlapped with the neighbouring steps' runs (timed from call to return)",
               "steps": e_steps, "ms_per_step": dt * 1e3 / e_steps,
               "single_call": {"value": s_units / dt1, "unit": UNIT, "steps": s_steps,
                               "ms_per_step": dt1 * 1e3 / s_steps,
                               "api": "fcm_run with pinned host buffers, one synchronous call per step"}}

    # device results kept for the precision report of the CPU-baseline leg
    keep = {"main": (Ud, Vd, r.iters, r.J)}

    # the other single-image workloads: the 200x200 and 1024x1024 phantoms
    # (on chip: latency-bound, no roofline) and the volume at the other
    # fuzzifiers (roofline as the main line)
    workloads = {}
    if not args.no_workloads:
        import phantom
        cases = [("phantom200", "phantom200", 2.0, 200), ("phantom1024", "phantom1024", 2.0, 50)]
        cases += [(f"volume256_m{mm:g}", "volume256", mm, 20) for mm in (1.5, 3.0) if mm != m]
        for key, name, mm, reps in cases:
            if name == "volume256":
                xw, u0w, xdw, u0dw = x, u0, xd, U0d
            else:
                xw, _, u0w, _ = phantom.single_image(name)
                xdw = torch.from_numpy(xw.astype(np.float32)).to(dev)
                u0dw = torch.from_numpy(u0w).to(dev)
            nw = xw.size
            Uw = torch.empty_like(u0dw)
            Vw = torch.empty(C, dtype=torch.float32, device=dev)
            for _ in range(args.warmup):
                rw = h.run(xdw, C, mm, EPS, MAX_ITER, U0=u0dw, U=Uw, V=Vw)
            torch.cuda.synchronize(dev)
            e0.record(stream)
            for _ in range(reps):
                rw = h.run(xdw, C, mm, EPS, MAX_ITER, U0=u0dw, U=Uw, V=Vw)
            e1.record(stream)
            torch.cuda.synchronize(dev)
            wms = e0.elapsed_time(e1) / reps
            ent = {"workload": workload_name(mm) if name == "volume256" else
                   f"{name}: {int(np.sqrt(nw))}x{int(np.sqrt(nw))} uint8 phantom as f32, C=4, m={mm:g}, eps=1e-5",
                   "n_pixels": nw, "m": mm, "runs": reps, "ms_per_run": wms, "images_per_s": 1e3 / wms,
                   "iters": rw.iters, "pixel_iter_per_s": nw * rw.iters / (wms / 1e3),
                   "us_per_iteration": wms * 1e3 / max(1, rw.iters)}
            if name == "volume256":
                ent["roofline"] = fp32_roofline(float(nw) * rw.iters, wms, C, mm, clocks.get("sm_mhz"))
            else:
                ent["bound"] = (f"latency: x ({4 * nw / 1e6:.1f} MB) sits in shared memory; "
                                "an iteration costs its dependent steps and its grid exchange")
            workloads[key] = ent
            keep[key] = (Uw, Vw, rw.iters, rw.J, xw, u0w, mm)

    # the same run on the grey-level histogram (fcm_run_hist), inputs resident
    hist = None
    if not args.no_hist:
        Uh = torch.empty_like(U0d)
        Vh = torch.empty(C, dtype=torch.float32, device=dev)
        for _ in range(args.warmup):
            rh = h.run_hist(xd, C, m, EPS, MAX_ITER, U0=U0d, U=Uh, V=Vh)
        hs = max(3, min(args.steps, 50))
        torch.cuda.synchronize(dev)
        e0.record(stream)
        for _ in range(hs):
            rh = h.run_hist(xd, C, m, EPS, MAX_ITER, U0=U0d, U=Uh, V=Vh)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        hms = e0.elapsed_time(e1) / hs
        hbytes = 2 * (4 + 4 * C) * n  # histogram + V^1 pass, U write
        hist = {"kernel": "fcm_run_hist: pixel passes for the histogram and the U write; "
                          "the iterations on 256 bins in one CTA",
                "ms_per_run": hms, "iters": rh.iters, "launches_per_run": rh.launches,
                "equivalent_pixel_iter_per_s": n * rh.iters / (hms / 1e3),
                "roofline": {"bound": "hbm", "achieved": hbytes / (hms / 1e3) / 1e9, "peak": peak, "unit": "GB/s",
                             "frac": hbytes / (hms / 1e3) / 1e9 / peak, "algorithmic_bytes_per_run": hbytes},
                "speedup_vs_pixel_path": (ms / args.steps) / hms}
        keep["histogram_domain"] = (Uh, Vh, rh.iters, rh.J)

    # the same run keeping no U between iterations (FCM_OPT_RECOMPUTE)
    recompute = None
    if not args.no_recompute:
        Ur = torch.empty_like(U0d)
        Vr = torch.empty(C, dtype=torch.float32, device=dev)
        for _ in range(args.warmup):
            rr = h.run(xd, C, m, EPS, MAX_ITER, U0=U0d, U=Ur, V=Vr, recompute=True)
        rs = max(3, min(args.steps, 50))
        torch.cuda.synchronize(dev)
        e0.record(stream)
        for _ in range(rs):
            rr = h.run(xd, C, m, EPS, MAX_ITER, U0=U0d, U=Ur, V=Vr, recompute=True)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        rms = e0.elapsed_time(e1) / rs
        rbytes = 2 * (4 + 4 * C) * n
        recompute = {"kernel": "k_fcm_run (FCM_OPT_RECOMPUTE insists on it)",
                     "ms_per_run": rms, "iters": rr.iters, "pixel_iter_per_s": n * rr.iters / (rms / 1e3),
                     "bound": "fp32 pipe",
                     "dram_bytes_per_run_algorithmic": rbytes,
                     "speedup_vs_pixel_path": (ms / args.steps) / rms,
                     "roofline": fp32_roofline(float(n) * rr.iters, rms, C, m, clocks.get("sm_mhz"))}
        keep["recompute"] = (Ur, Vr, rr.iters, rr.J)

    # multi-feature FCM on a 3-channel 2048^2 phantom (shared layout, per-channel
    # contrasts and noise), inputs resident
    multi = None
    if not args.no_multi:
        import phantom
        xm, _ = phantom.multichannel2d(5, 2048, 2048, 8.0, [(0.0, 40.0, 110.0, 150.0), (0.0, 150.0, 90.0, 60.0),
                                                            (10.0, 200.0, 120.0, 80.0)])
        nm = xm.shape[1]
        xmd = torch.from_numpy(xm.astype(np.float32)).to(dev)
        u0m = torch.from_numpy(phantom.dirichlet_u0((5, 3), C, nm)).to(dev)
        Um = torch.empty((C, nm), dtype=torch.float32, device=dev)
        for _ in range(args.warmup):
            rm = h.run_multi(xmd, C, m, EPS, MAX_ITER, U0=u0m, U=Um)
        ms_ = max(3, min(args.steps, 20))
        torch.cuda.synchronize(dev)
        e0.record(stream)
        for _ in range(ms_):
            rm = h.run_multi(xmd, C, m, EPS, MAX_ITER, U0=u0m, U=Um)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        mms = e0.elapsed_time(e1) / ms_
        multi = {"workload": "3-channel 2048x2048 phantom, C=4, m=2, eps=1e-5", "channels": 3, "n_pixels": nm,
                 "ms_per_run": mms, "iters": rm.iters, "pixel_iter_per_s": nm * rm.iters / (mms / 1e3),
                 "roofline": issue_roofline("profiles/fcm_multi_3ch_2048.md",
                                            ["paper_1601_00072_gb300/csrc/fcm_multi_inst.cu",
                                             "paper_1601_00072_gb300/csrc/fcm_device.cuh",
                                             "paper_1601_00072_gb300/csrc/fcm_multi.h"],
                                            mms, rm.iters, clocks.get("sm_max_mhz"))}
        keep["multi_feature"] = (xm, u0m.cpu().numpy(), Um, rm)

    # the paper's quantitative score (Dice per tissue class, Sec. 5.2) of the
    # timed run's segmentation against the phantom's generator labels
    labd = torch.from_numpy(lab.astype(np.uint8)).to(dev)
    dsc, _ = h.dsc(Ud, labd, n_classes=C, V=Vd)
    dsc_line = {"classes": ["background", "CSF", "GM", "WM"], "dsc": [round(float(d), 6) for d in dsc],
                "truth": "phantom generator labels", "cluster_to_class": "by ascending center"}

    out = {
        "metric": METRIC,
        "value": value,
        "unit": UNIT,
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": ms / args.steps,
        "step_ms": {"mean": statistics.mean(per_step), "median": statistics.median(per_step),
                    "min": min(per_step), "max": max(per_step)},
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": workload_name(m),
                   "n_pixels": n, "iters_per_step": statistics.median(iters),
                   "parallelism": f"replicas x{world}",
                   "l2": "working set 603 MB > 129 MB L2; no flush"},
        "gpu_launches": launches,
        "roofline": dict(fp32_roofline(units_local, ms_local, C, m, clocks.get("sm_mhz")), traffic=traffic,
                         kernel="k_fcm_run: one cooperative launch per step (pass 0 reads x and U0; the "
                                "iterations read x from shared memory and the L2; U is written once)",
                         algorithmic_bytes_per_step=bytes_local / args.steps,
                         hbm={"achieved": hbm_gbs, "peak": peak, "unit": "GB/s", "frac": hbm_gbs / peak,
                              "peak_source": f"{peak_kind} copy bandwidth"}),
        "clocks": clocks,
        "e2e": e2e,
        "histogram_domain": hist,
        "recompute": recompute,
        "segmentation_dsc": dsc_line,
        "multi_feature": multi,
        "other_workloads": workloads,
    }
    if not args.no_batched:
        out["batched"], keep["batched"] = bench_batched(h, dev, max(3, min(args.steps, 20)), 3, keep_results=True)
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline_leg(x, u0, m, keep, out)
    h.close()
    if rank == 0:
        print(json.dumps(out))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def bench_reference(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    x, u0 = load_workload(args.m)
    xs, us, desc = cpu_sample(x, u0)
    # a smaller slab per step keeps --steps K --warmup W within minutes
    plane = 256 * 256
    xs, us = xs[:4 * plane], np.ascontiguousarray(us[:, :4 * plane])
    import oracle
    it = 10

    def step():
        return oracle.fcm(xs.astype(np.float64), C, args.m, 0.0, it, U0=us, want_U=False)

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    units = 0
    for _ in range(args.steps):
        r = step()
        units += xs.size * r["iters"]
    dt = time.perf_counter() - t0
    value = units / dt
    sample = f"262,144 voxels (slices z=120..123) x {it} iterations per step"
    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": dt * 1e3 / args.steps, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "impl": "reference",
           "config": {"workload": workload_name(args.m), "n_pixels": 256 ** 3,
                      "sample": "each step: 262,144 voxels (slices z=120..123) x 10 iterations of the FP64 oracle"},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out))


def main():
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--m", type=float, default=2.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-batched", action="store_true", help="skip the cold versus warm batch measurement")
    ap.add_argument("--no-hist", action="store_true", help="skip the histogram-domain measurement")
    ap.add_argument("--no-recompute", action="store_true", help="skip the U-free (recompute) measurement")
    ap.add_argument("--no-multi", action="store_true", help="skip the multi-feature measurement")
    ap.add_argument("--no-workloads", action="store_true",
                    help="skip the 200x200 and 1024x1024 phantoms and the volume at the other fuzzifiers")
    ap.add_argument("--batched-only", action="store_true",
                    help="only the cold versus warm batch measurement, printed as its own JSON object "
                         "(a profiling aid; not the benchmark line)")
    ap.add_argument("--batch-slices", type=int, default=512,
                    help="with --batched-only: the first N slices of the batch (a small case for profilers)")
    ap.add_argument("--batch-plan", default=None,
                    help='with --batched-only: a fixed launch plan instead of the autotuner, as JSON, '
                         'e.g. \'{"block": 256, "cluster": 4, "big": 16384}\'')
    ap.add_argument("--variant", choices=["tma", "ldg"], default="tma",
                    help="pass kernel: TMA-fed ring (default) or plain loads")
    ap.add_argument("--no-graph", action="store_true",
                    help="launch the same pass kernels from a host loop instead of the CUDA graph "
                         "WHILE node (for profilers that cannot see kernels inside conditional graphs)")
    args = ap.parse_args()
    if args.warmup < 3 and args.impl == "ours" and not os.environ.get("FCM_BENCH_ALLOW_SHORT"):
        print("warning: fewer than 3 warm-up steps", file=sys.stderr)
    if args.impl == "reference":
        bench_reference(args)
    elif args.batched_only:
        import torch
        from paper_1601_00072_gb300 import _build
        _build.build()
        from paper_1601_00072_gb300.fcm import FCM
        h = FCM(0)
        plan = json.loads(args.batch_plan) if args.batch_plan else None
        print(json.dumps(bench_batched(h, torch.device("cuda", 0), max(1, args.steps), args.warmup, plan,
                                       n_slices=args.batch_slices)))
        h.close()
    else:
        bench_ours(args)


if __name__ == "__main__":
    main()
