#!/usr/bin/env python3
"""Benchmark of the DGSEM hot path: rhs DOF-evaluations per second (1/PID).

One step = one Carpenter-Kennedy LSRK time step of the 3D compressible Euler
DGSEM: the CFL time step (a wave-speed reduction and the dt formula, on the
device) and five stages, each a surface-flux kernel and the flux-differencing
volume kernel with lifting and the stage update fused into its epilogue; the
step is replayed as a CUDA graph. The metric counts (N+1)^3 nodes x
elements x 5 rhs evaluations per step over the wall time (the paper's
performance index PID = time / (steps 5 elements (N+1)^3), inverted).

Default workload: 3D Euler, N=3, 64^3 periodic elements on [-1,1]^3, density
wave rho = 1 + 0.98 sin(pi(x+y+z)), v = (0.1,0.2,0.3), p = 20, plus seeded
uniform 1e-2 noise on rho, v and p (seed 0); Ranocha EC volume flux, LLF
surface flux. The FP64 path gives `value`; the FP32 kernels (FP64 state and
RK accumulation) are timed on the same state and reported under "fp32".

`--impl reference` times the plain CPU oracle on a bounded sample of the
same workload instead.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "rhs DOF-evals/s (1/PID) 3D Euler N=3, FP32 vs FP64 at stated error; % of FP64 peak"
UNIT = "DOF-rhs-evals/s"

WORKLOADS = {
    "euler3d_n3_64cubed_noisy_wave": dict(d=3, N=3, ne=64, noise=1e-2),
    "euler3d_n3_32cubed_wave": dict(d=3, N=3, ne=32, noise=0.0),
    "euler3d_n7_24cubed_noisy_wave": dict(d=3, N=7, ne=24, noise=1e-2),
}
DEFAULT_WORKLOAD = "euler3d_n3_64cubed_noisy_wave"

# Vector peaks: measured on the device at start-up by the library's FMA
# throughput probe (dg_measure_peaks); the nominal figures (2 DFMA and 128
# FFMA lanes per clock per SM at 2070 MHz) are reported beside them.
NOMINAL_SM_MHZ = 2070.0


def nominal_peaks(sms):
    return {"fp64_tflops": sms * 2 * 2 * NOMINAL_SM_MHZ * 1e6 / 1e12,
            "fp32_tflops": sms * 128 * 2 * NOMINAL_SM_MHZ * 1e6 / 1e12}


PEAKS = {}


def measured_hbm_gbs():
    """The copy bandwidth of this machine's GPUs (MEASURED_PEAKS.json), or None."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return float(json.load(fh)["hbm_gbs"])
    except (OSError, ValueError, KeyError, TypeError):
        return None


def measured_peaks():
    """FP64/FP32 FMA throughput and SM count, measured once per process."""
    if not PEAKS:
        from paper_2108_06476_gb300 import measure_peaks
        PEAKS.update(measure_peaks())
    return PEAKS


def cpu_model():
    """The host CPU's model name (lscpu, else /proc/cpuinfo)."""
    try:
        r = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=30)
        for ln in r.stdout.splitlines():
            if ln.startswith("Model name:"):
                return ln.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    try:
        with open("/proc/cpuinfo") as fh:
            for ln in fh:
                if ln.lower().startswith(("model name", "cpu model")):
                    return ln.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return platform.processor() or platform.machine()


OP_COUNTS = os.path.join(ROOT, "tests", "golden", "op_counts.json")


def counted_ops(workload):
    """The algorithmic operations per node of the volume kernel for a
    configured workload, as counted by the oracle's operation-counting build
    (written by tests/golden/make_op_counts.py): None if not recorded."""
    try:
        with open(OP_COUNTS) as fh:
            return json.load(fh)["workloads"].get(workload)
    except (OSError, ValueError, KeyError):
        return None


def volume_flops_per_node(d, N):
    """A hand count of the flops per node of the rhs volume kernel (Ranocha
    flux; log, division and square root count as one flop each): pairs per
    node d N / 2, each 46 + 5d flops of flux and 4 (d+2) of accumulation;
    prologue 3d + 3; lifting 4 d (d+2) / (N+1). Reported beside the oracle's
    counted figure, which the roofline uses."""
    pair = 46 + 5 * d + 4 * (d + 2)
    return d * N / 2 * pair + 3 * d + 3 + 4 * d * (d + 2) / (N + 1)


KERNEL_SOURCES = ("dg_device.cuh", "dg_fixed.cuh", "dg_fixed_tables.cuh", "dg_fixed_volume.cuh",
                  "dg_fixed_face.cuh", "dg_rhs_kernels.cuh", "dg_rhs_inst.cu")


def _code_only(text):
    """Source text without comments and whitespace (a comment edit does not
    change a kernel)."""
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    text = re.sub(r"//[^\n]*", " ", text)
    return re.sub(r"\s+", "", text)


MHD_KERNEL_SOURCES = ("dg_device.cuh", "dg_fixed.cuh", "dg_fixed_tables.cuh", "dg_fixed_face.cuh",
                      "dg_rhs_kernels.cuh", "dg_mhd_weak.cuh", "dg_mhd.cu")


def source_sha(files=KERNEL_SOURCES):
    """Hash of the code (comments and whitespace removed) of the sources that
    define a family of kernels (the Euler rhs kernels by default): a
    committed ncu figure is only used while it is unchanged."""
    h = hashlib.sha1()
    csrc = os.path.join(ROOT, "paper_2108_06476_gb300", "csrc")
    for fn in files:
        with open(os.path.join(csrc, fn)) as fh:
            h.update(fn.encode() + _code_only(fh.read()).encode())
    return h.hexdigest()[:12]


def ncu_record(key, field):
    """A per-node figure of a kernel from a committed ncu summary (DRAM bytes,
    counted flops), or None when the kernels changed since that capture."""
    path = os.path.join(ROOT, "profiles", "dram_traffic.json")
    try:
        with open(path) as fh:
            rec = json.load(fh).get(key)
    except (OSError, ValueError):
        return None
    if not rec:
        return None
    files = tuple(rec.get("sources", KERNEL_SOURCES))
    if rec.get("src_sha") != (source_sha() if files == KERNEL_SOURCES else source_sha(files)):
        return None
    return rec.get(field)


def ncu_traffic(key):
    return ncu_record(key, "bytes_per_node")


class ClockSampler:
    """Samples nvidia-smi SM clocks and throttle reasons during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.lines = []
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[4:8]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


def make_state(spec, xi, seed=0):
    from paper_2108_06476_gb300 import workloads as W
    d, N, ne = spec["d"], spec["N"], spec["ne"]
    n = (ne,) * d
    dom = W.box(d)
    if spec["noise"] > 0:
        return W.noisy_density_wave(d, N, n, dom, xi, seed=seed, noise=spec["noise"])
    return W.density_wave(d, N, n, dom, xi)


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def run_reference(args, spec, world, rank):
    """The plain CPU oracle on a bounded sample of the workload's elements:
    each step = 5 x (oracle rhs on the sample + oracle stage update of the
    sample's values)."""
    if rank != 0:
        return
    import numpy as np
    import oracle
    oracle.build()
    d, N, ne = spec["d"], spec["N"], spec["ne"]
    n = (ne,) * d
    from paper_2108_06476_gb300 import workloads as W
    dom = W.box(d)
    xi, _ = oracle.lgl(N)
    u = make_state(spec, xi)
    P, nv = (N + 1) ** d, d + 2
    nelem = ne ** d
    cores = os.cpu_count() or 1
    # size the sample: about 1.5 s of oracle work per step
    probe = np.arange(0, nelem, max(1, nelem // 256))[:256]
    du = np.zeros_like(u)
    t = time.perf_counter()
    oracle.rhs(d, N, n, dom, u, elems=probe, out=du)
    per_elem = (time.perf_counter() - t) / len(probe)
    count = int(min(nelem, max(64, 0.3 / max(per_elem, 1e-9))))
    rng = np.random.default_rng(1)
    elems = np.sort(rng.choice(nelem, size=count, replace=False))
    A, B, _ = oracle.lsrk_coefficients()
    uu = u.reshape(nelem, nv * P)
    k = np.zeros((count, nv * P))
    dt = 1e-5

    def step():
        for s in range(5):
            oracle.rhs(d, N, n, dom, u, elems=elems, out=du)
            us = np.ascontiguousarray(uu[elems])
            ds = np.ascontiguousarray(du.reshape(nelem, nv * P)[elems])
            oracle.rk_stage(us, k, ds, A[s], B[s], dt)
            uu[elems] = us

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        step()
    el = time.perf_counter() - t0
    value = count * P * 5 * args.steps / el
    sample = (f"{count} of {nelem} elements ({count * P} of {nelem * P} nodes) of {args.workload}, "
              f"5 rhs + 5 stage updates per step")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": el / args.steps * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": args.workload, "d": d, "N": N, "elements_per_dim": ne,
                       "volume_flux": "ranocha", "surface_flux": "llf"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ensemble(args, timed, rank, checks):
    """The seeded 48-member ensemble advanced with one launch per stage and a
    CUDA-graph step, after the autotuner picked the CTA shape; FP64 and FP32.
    Records one stage's rhs of every member on a few sampled elements for the
    oracle check of the baseline leg."""
    import numpy as np
    import torch
    from paper_2108_06476_gb300 import Ensemble, lgl_nodes, RK_B, workloads as W
    mem = W.ensemble(n_sims=48, seed=rank)
    u0h = W.ensemble_state(mem, lambda N: lgl_nodes(N)[0])
    u0 = torch.from_numpy(u0h).cuda()
    out = {"workload": f"48 periodic 3D density waves (seed {rank}), N in {{3,4,5}}, "
                       "n in [8,24]", "members": len(mem)}
    k = max(1, min(args.steps, 5))
    for prec in ("fp64", "fp32"):
        E = Ensemble([m.N for m in mem], [m.n[0] for m in mem], precision=prec)
        u = u0.clone()
        tmp = torch.empty_like(u)
        threads, per_sm, stage_ms = E.tune(u, tmp)
        grid = E.get_block()[2]
        # one stage with a large dt recovers every member's rhs (checked
        # against the oracle on sampled elements in the baseline leg)
        big = 1.0e6
        E.set_dt(np.full(E.n_sims, big))
        E.stage(u, tmp, 0)
        E.rk_reset()
        got = (tmp.cpu().numpy() - u0h) / (RK_B[0] * big)
        samples = []
        for s_, m in enumerate(mem):
            ne, P = m.n[0] ** 3, (m.N + 1) ** 3
            el = np.unique(np.concatenate([[0, ne - 1], np.random.default_rng(s_).choice(
                ne, size=min(ne, 12), replace=False)]))
            part = got[E.offsets[s_]:E.offsets[s_ + 1]].reshape(ne, 5, P)[el]
            samples.append((m, u0h[E.offsets[s_]:E.offsets[s_ + 1]], el, part))
        checks.append(("ensemble", prec, samples))
        by_tpl = None
        if prec == "fp64":
            # one stage in each threads-per-line mode at the tuned CTA shape
            tuned_pair = E.pair_parallel
            by_tpl = {}
            for mode, name in ((False, "1"), (True, "one per node pair")):
                E.pair_parallel = mode
                E.stage(u, tmp, 1)
                by_tpl[name] = timed(lambda: E.stage(u, tmp, 1))
            E.pair_parallel = tuned_pair
            E.rk_reset()
        for _ in range(args.warmup):
            E.step(u, cfl=0.5, graph=True)
        ms = timed(lambda: [E.step(u, cfl=0.5, graph=True) for _ in range(k)])
        E.check()
        out[prec] = {"value": E.n_nodes * 5 * k / (ms / 1e3), "unit": UNIT,
                     "ms_per_step": ms / k, "tuned_threads": threads,
                     "tuned_ctas_per_sm": per_sm, "ctas_launched": grid,
                     "tuned_threads_per_line": ("one per node pair" if E.pair_parallel
                                                else 1),
                     "tuner_searched": {"threads_per_cta": [64, 96, 128],
                                        "ctas_per_sm": [1, 2, 3, 4, 6],
                                        "threads_per_line": ([1, "one per node pair"]
                                                             if prec == "fp64" else [1])},
                     "tuned_stage_ms": stage_ms,
                     "stage_ms_by_threads_per_line": by_tpl,
                     "stage_launches_per_step": 5}
        # the step's algorithmic work: every member's nodes x the operations
        # per node of its degree (oracle operation counts) x 5 stages
        per_n = {N: counted_ops(f"ensemble_member_n{N}") for N in (3, 4, 5)}
        if all(per_n.values()):
            ops = 5 * sum(m.n[0] ** 3 * (m.N + 1) ** 3 * per_n[m.N]["volume_fused_per_node"]
                          for m in mem)
            tf = ops / (ms / k / 1e3) / 1e12
            peak = measured_peaks()["fp64_tflops" if prec == "fp64" else "fp32_tflops"]
            out[prec]["step_tflops"] = tf
            out[prec]["step_frac_of_peak"] = tf / peak
            out[prec]["ops_source"] = ("oracle operation counts per degree "
                                       "(tests/golden/op_counts.json, ensemble_member_n*), "
                                       "whole step time, measured peak of the precision")
        out["nodes"] = E.n_nodes
        del E, u, tmp
    return out


def _sample_elements(nelem, count, seed):
    import numpy as np
    if nelem <= count:
        return np.arange(nelem)
    rng = np.random.default_rng(seed)
    return np.unique(np.concatenate([[0, nelem - 1], rng.choice(nelem, size=count,
                                                                  replace=False)]))


def graph_ms(fn, timed):
    """Record fn (library calls on the current stream) as one CUDA graph and
    time a replay; None if the capture is refused."""
    import torch
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    try:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(stream):
            fn()  # warm-up on the capture stream
            torch.cuda.synchronize()
            with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
                fn()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        return timed(lambda: g.replay())
    except RuntimeError:
        return None


def run_configs(args, timed, checks):
    """rhs-only rates (50 back-to-back dg_rhs calls, FP64 and FP32 kernels)
    and the fused-step rate (FP64, CUDA-graph CFL steps) of the other
    configured cases: 2D 16^2 N=3 and 3D 32^3 N=3 density waves, 3D 24^3 N=7
    noisy density wave. Each rhs is recorded on sampled elements for the
    oracle check of the baseline leg."""
    import torch
    from paper_2108_06476_gb300 import Mesh, lgl_nodes, workloads as W
    out = {}
    for name, d, N, ne, noisy in (("euler2d_n3_16sq_density_wave", 2, 3, 16, False),
                                  ("euler3d_n3_32cubed_density_wave", 3, 3, 32, False),
                                  ("euler3d_n7_24cubed_noisy_wave", 3, 7, 24, True)):
        n = (ne,) * d
        xi, _ = lgl_nodes(N)
        gen = W.noisy_density_wave if noisy else W.density_wave
        uh = gen(d, N, n, W.box(d), xi)
        u0 = torch.from_numpy(uh).cuda()
        row = {"nodes": ne ** d * (N + 1) ** d}
        elems = _sample_elements(ne ** d, 200 if N < 7 else 40, seed=ne)
        for prec in ("fp64", "fp32"):
            m = Mesh(d, N, n, precision=prec)
            du = m.empty_rhs()
            m.rhs(u0, du)
            nv, P = d + 2, (N + 1) ** d
            checks.append(("configs", (name, f"rhs_{prec}"), (d, N, n, uh, elems, du.double()
                          .cpu().numpy().reshape(-1, nv, P)[elems])))
            ms = timed(lambda: [m.rhs(u0, du) for _ in range(50)])
            row[f"rhs_{prec}"] = row["nodes"] * 50 / (ms / 1e3)
            # the same 50 calls recorded once as a CUDA graph and replayed:
            # the kernels' rate without the host's per-call cost (small meshes)
            ms_g = graph_ms(lambda: [m.rhs(u0, du) for _ in range(50)], timed)
            if ms_g is not None:
                row[f"rhs_{prec}_graph"] = row["nodes"] * 50 / (ms_g / 1e3)
            if prec == "fp64":
                u = u0.clone()
                for _ in range(3):
                    m.step_cfl(u, cfl=0.5, graph=True)
                ms = timed(lambda: [m.step_cfl(u, cfl=0.5, graph=True) for _ in range(10)])
                row["step_fp64"] = row["nodes"] * 5 * 10 / (ms / 1e3)
            m.check()
            del m, du
        out[name] = row
    out["unit"] = UNIT
    return out


def run_vjp(args, timed):
    """dg_rhs_vjp (the hand-written vector-Jacobian product) on the VJP
    configuration: 3D N=4, 16^3 periodic elements, noisy density wave, N(0,1)
    cotangent; FP64 and FP32 Jacobians, 20 back-to-back calls each."""
    import torch
    from paper_2108_06476_gb300 import Mesh, lgl_nodes, workloads as W
    d, N, n = 3, 4, (16, 16, 16)
    xi, _ = lgl_nodes(N)
    u = torch.from_numpy(W.noisy_density_wave(d, N, n, W.box(d), xi, seed=0)).cuda()
    w = torch.from_numpy(W.gaussian(u.numel(), seed=1)).cuda()
    out = {"workload": "VJP of the 3D Euler rhs, N=4, 16^3 periodic elements, noisy density "
                       "wave, N(0,1) cotangent", "unit": UNIT}
    reps = 20
    for prec in ("fp64", "fp32"):
        m = Mesh(d, N, n, precision=prec)
        ub = torch.empty_like(u)
        m.rhs_vjp(u, w, ub)
        ms = timed(lambda: [m.rhs_vjp(u, w, ub) for _ in range(reps)])
        du = m.empty_rhs()
        m.rhs(u, du)
        ms_rhs = timed(lambda: [m.rhs(u, du) for _ in range(reps)])
        out[prec] = {"value": m.n_nodes * reps / (ms / 1e3), "ms_per_vjp": ms / reps,
                     "vjp_over_rhs_time": ms / ms_rhs}
        m.check()
        del m, ub, du
    out["nodes"] = 16 ** 3 * (N + 1) ** 3
    return out


def oracle_config_rates(seconds=1.0):
    """The oracle's rhs rate (OpenMP on all host cores, and one thread) on a
    bounded sample of each configured case: elements sampled for about
    `seconds` each (the oracle's per-node work does not depend on the mesh
    size, only on d and N)."""
    import numpy as np
    import oracle
    from paper_2108_06476_gb300 import workloads as W
    oracle.build()
    out = {}
    for name, d, N, ne, noisy in (("euler2d_n3_16sq_density_wave", 2, 3, 16, False),
                                  ("euler3d_n3_32cubed_density_wave", 3, 3, 32, False),
                                  ("euler3d_n3_64cubed_noisy_wave", 3, 3, 64, True),
                                  ("euler3d_n7_24cubed_noisy_wave", 3, 7, 24, True)):
        n = (ne,) * d
        xi, _ = oracle.lgl(N)
        gen = W.noisy_density_wave if noisy else W.density_wave
        u = gen(d, N, n, W.box(d), xi)
        du = np.zeros_like(u)
        nelem, P = ne ** d, (N + 1) ** d
        row = {}
        for key, threads in (("all_cores", 0), ("single_core", 1)):
            probe = np.arange(min(nelem, 64))
            t = time.perf_counter()
            oracle.rhs(d, N, n, W.box(d), u, elems=probe, out=du, nthreads=threads)
            per = (time.perf_counter() - t) / len(probe)
            count = int(min(nelem, max(16, seconds / max(per, 1e-9))))
            elems = np.sort(np.random.default_rng(5).choice(nelem, size=count, replace=False))
            best = None
            for _ in range(3):
                t = time.perf_counter()
                oracle.rhs(d, N, n, W.box(d), u, elems=elems, out=du, nthreads=threads)
                el = time.perf_counter() - t
                best = el if best is None else min(best, el)
            row[key] = count * P / best
        oracle.rhs(d, N, n, W.box(d), u, elems=np.arange(1), out=du,
                   nthreads=os.cpu_count() or 1)  # restore the thread team
        out[name] = row
    out["unit"] = UNIT
    out["sample"] = "best of 3 oracle rhs evaluations over about 1 s of sampled elements"
    return out


def oracle_checks(line, checks, headline):
    """The baseline leg's accuracy record: the oracle's rhs on the sampled
    elements of every recorded GPU rhs (headline FP64/FP32, the configured
    cases, the 48 ensemble members), as relative L2 errors beside the rates."""
    import numpy as np
    import oracle
    from paper_2108_06476_gb300 import workloads as W
    oracle.build()

    def rel(a, b):
        return float(np.linalg.norm(a - b) / np.linalg.norm(b))

    d, N, n, uh, elems, gpu = headline
    nv, P = d + 2, (N + 1) ** d
    ref = oracle.rhs(d, N, n, W.box(d), uh, elems=elems).reshape(-1, nv, P)[elems]
    line["rhs_rel_l2_vs_oracle"] = {prec: rel(g, ref) for prec, g in gpu.items()}
    line["rhs_rel_l2_vs_oracle"]["sample"] = f"{len(elems)} of {int(np.prod(n))} elements"
    if line.get("fp32") is not None:
        line["fp32"]["rel_l2_vs_oracle"] = line["rhs_rel_l2_vs_oracle"]["fp32"]
    for kind, key, data in checks:
        if kind == "configs":
            name, field = key
            dd, NN, nn, u, el, g = data
            r = oracle.rhs(dd, NN, nn, W.box(dd), u, elems=el).reshape(-1, dd + 2,
                                                                      (NN + 1) ** dd)[el]
            if line.get("configs"):
                line["configs"][name][f"{field}_rel_l2_vs_oracle"] = rel(g, r)
                line["configs"][name]["oracle_sample"] = f"{len(el)} of {int(np.prod(nn))} elements"
        elif kind == "ensemble" and line.get("ensemble"):
            errs, cond, kappas = [], [], []
            for m, u, el, g in data:
                ne, PP = m.n[0] ** 3, (m.N + 1) ** 3
                r = oracle.rhs(3, m.N, m.n, W.box(3), u, elems=el).reshape(ne, 5, PP)[el]
                errs.append(rel(g, r))
                # the FP32 bar's scale: max(|du|, |sum_d |du_d|| / 3) from the
                # oracle's direction split (|du| unless the directions cancel)
                mag = sum(np.abs(oracle.rhs(3, m.N, m.n, W.box(3), u, elems=el, directions=[k])
                                 .reshape(ne, 5, PP)[el]) for k in range(3))
                kappas.append(float(np.linalg.norm(mag) / np.linalg.norm(r)))
                scale = max(np.linalg.norm(r), np.linalg.norm(mag) / 3.0)
                cond.append(float(np.linalg.norm(g - r) / scale))
            line["ensemble"][key]["rel_l2_vs_oracle"] = {
                "max_over_members": max(errs), "median": float(np.median(errs)),
                "max_over_members_vs_direction_scale": max(cond),
                "kappa_max": max(kappas),
                "sample": "2 corner + 12 random elements of each of the 48 members",
                "direction_scale": "error / max(|du|, |sum_d |du_d||/3), du_d the oracle's "
                                   "per-direction parts; kappa = |sum_d |du_d|| / |du|"}


def run_curved(args, timed):
    """The paper's PID setup (Sec. 3.1) on the GPU: the warped periodic box
    [-1,1]^3 of 4^3 elements, the manufactured solution with its source
    terms, CFL 0.5 steps (device time step, CUDA graph), degrees 3..7, for the
    flux-differencing solver (Ranocha volume and surface flux) and the
    weak-form solver (central volume flux, HLL surface flux); PID =
    time / (steps * 5 * nodes). Plus the same operator on 64^3 warped
    elements (N = 3, flux differencing) for throughput."""
    import torch
    from paper_2108_06476_gb300 import Mesh, lgl_nodes, workloads as W
    out = {"workload": "warped periodic box [-1,1]^3 (warp 0.15), manufactured solution "
                       "with source terms, CFL 0.5, CUDA-graph steps", "pid_4cubed": {}}
    k = max(1, min(args.steps, 5)) * 20
    for solver, vf, sf in (() if args.no_pid else
                           (("flux_differencing", "ranocha", "ranocha"),
                            ("weak_form", "central", "hll"))):
        rows = {}
        for N in range(3, 8):
            n = (4, 4, 4)
            m = Mesh(3, N, n, warp=0.15, volume_flux=vf, surface_flux=sf)
            m.set_source("manufactured")
            xi, _ = lgl_nodes(N)
            u = torch.from_numpy(W.manufactured_state(
                W.warped_node_coordinates(N, n, xi, 0.15), 0.0)).cuda()
            for _ in range(max(3, args.warmup)):
                m.step_cfl(u, cfl=0.5, graph=True)
            ms = timed(lambda: [m.step_cfl(u, cfl=0.5, graph=True) for _ in range(k)])
            m.check()
            rows[str(N)] = {"pid_s": ms / 1e3 / (k * 5 * m.n_nodes), "ms_per_step": ms / k,
                            "nodes": m.n_nodes}
            del m, u
        out["pid_4cubed"][solver] = rows
    ne = args.curved_elements
    n = (ne, ne, ne)
    m = Mesh(3, 3, n, warp=0.15)
    m.set_source("manufactured")
    xi, _ = lgl_nodes(3)
    u = torch.from_numpy(W.manufactured_state(
        W.warped_node_coordinates(3, n, xi, 0.15), 0.0)).cuda()
    for _ in range(max(3, args.warmup)):
        m.step_cfl(u, cfl=0.5, graph=True)
    kk = max(1, min(args.steps, 5))
    ms = timed(lambda: [m.step_cfl(u, cfl=0.5, graph=True) for _ in range(kk)])
    m.check()
    out[f"warped_{ne}cubed_n3"] = {"value": m.n_nodes * 5 * kk / (ms / 1e3), "unit": UNIT,
                                   "ms_per_step": ms / kk, "nodes": m.n_nodes}
    return out


def mhd_volume_flops_per_node(N):
    """Algorithmic FP64 flops per node of the MHD volume kernel (rhs only, a
    fused multiply-add counted as two, a reciprocal as one): 28 for the
    node's primitives, 14 for the Powell term, and per direction 20 for the
    flux, 16 (N+1) for the eight D-row products (seven flux components and
    B_n), and the lifting (26 flops) at the 2 of N+1 line nodes on a face."""
    return 42 + 3 * (20 + 16 * (N + 1) + 52 / (N + 1))


def run_mhd(args, timed, kernel_ms):
    """3D ideal MHD with the Powell term (the Alfven-wave setting of
    Sec. 3.1) on the GPU: the circularly polarised Alfven wave on ne^3
    elements of degree 3, CFL 0.5 steps (device time step, CUDA graph): the
    paper's two solvers, the weak form with HLL faces (and LLF for
    comparison) and EC flux differencing with EC faces, with the kernel
    times of one rhs."""
    import torch
    from paper_2108_06476_gb300 import Mesh, lgl_nodes, workloads as W
    ne, N = args.mhd_elements, 3
    n = (ne, ne, ne)
    xi, _ = lgl_nodes(N)
    u0 = torch.from_numpy(W.alfven_wave(N, n, xi, 0.0)).cuda()
    kk = max(1, min(args.steps, 10))
    out = {}
    for key, vf, sf in (("hll", "central", "hll"), ("llf", "central", "llf"), ("ec", "ec", "ec")):
        m = Mesh(3, N, n, equations="mhd", surface_flux=sf, volume_flux=vf)
        u = u0.clone()
        du = m.empty_rhs()
        for _ in range(max(3, args.warmup)):
            m.step_cfl(u, cfl=0.5, graph=True)
        ms = timed(lambda: [m.step_cfl(u, cfl=0.5, graph=True) for _ in range(kk)])
        m.check()
        M = m.n_nodes
        row = {"value": M * 5 * kk / (ms / 1e3), "unit": UNIT, "ms_per_step": ms / kk,
               "kernels_ms": {"volume_fused_stage": kernel_ms(m, u, du, 6),
                              "volume_rhs_only": kernel_ms(m, u, du, 2),
                              "surface": kernel_ms(m, u, du, 1)}}
        out[key] = row
        del m, u, du
    # PID sweeps on 4^3 elements, N = 3..7, both solvers: the warped box of
    # the paper's MHD PID runs, and the Cartesian mesh for comparison
    pid, pid_warped = {}, {}
    if not args.no_pid:
        kp = max(1, min(args.steps, 5)) * 20
        for (key, vf, sf), warp in [(c, w) for w in (None, 0.15) for c in (
                ("weak_form_hll", "central", "hll"), ("ec_flux_differencing", "ec", "ec"))]:
            rows = {}
            for Np in range(3, 8):
                np_ = (4, 4, 4)
                xi_p, _ = lgl_nodes(Np)
                mp = Mesh(3, Np, np_, equations="mhd", surface_flux=sf, volume_flux=vf, warp=warp)
                Xp = (W.node_coordinates(3, Np, np_, W.box(3), xi_p) if warp is None
                      else W.warped_node_coordinates(Np, np_, xi_p, warp))
                up = torch.from_numpy(W.alfven_wave_at(Xp, 0.0)).cuda()
                for _ in range(max(3, args.warmup)):
                    mp.step_cfl(up, cfl=0.5, graph=True)
                msp = timed(lambda: [mp.step_cfl(up, cfl=0.5, graph=True) for _ in range(kp)])
                mp.check()
                rows[str(Np)] = {"pid_s": msp / 1e3 / (kp * 5 * mp.n_nodes),
                                 "ms_per_step": msp / kp, "nodes": mp.n_nodes}
                del mp, up
            (pid if warp is None else pid_warped)[key] = rows
    fl = mhd_volume_flops_per_node(N)
    vol = out["hll"]["kernels_ms"]["volume_rhs_only"]
    ach = fl * M / (vol / 1e3) / 1e12
    traffic = ncu_traffic("fp64_mhd_volume_n3")
    counted_node = ncu_record("fp64_mhd_volume_n3", "fp64_flops_executed_per_node")
    return {"workload": f"3D ideal MHD, circularly polarised Alfven wave, {ne}^3 elements, "
                        "N = 3, weak form + Powell term, HLL faces, CFL 0.5, CUDA-graph steps",
            "value": out["hll"]["value"], "unit": UNIT, "ms_per_step": out["hll"]["ms_per_step"],
            "nodes": M, "state_mb": M * 8 * 8 / 1e6, "kernels_ms": out["hll"]["kernels_ms"],
            "llf": out["llf"],
            "ec_flux_differencing": out["ec"],
            "pid_4cubed_warped": pid_warped,
            "pid_4cubed_cartesian": pid,
            "roofline": {"bound": "alu", "kernel": "mhd_volume_weak_kernel (rhs only)",
                         "flops_per_node": fl, "achieved": ach,
                         "peak": measured_peaks()["fp64_tflops"],
                         "peak_source": "measured (dg_measure_peaks, FP64 FMA probe)",
                         "unit": "TFLOP/s", "frac": ach / measured_peaks()["fp64_tflops"],
                         "traffic": None if traffic is None else traffic * M,
                         "counted": None if counted_node is None else {
                             "flops_per_node": counted_node,
                             "achieved": counted_node * M / (vol / 1e3) / 1e12,
                             "frac": counted_node * M / (vol / 1e3) / 1e12
                             / measured_peaks()["fp64_tflops"]}}}


def mhd_cpu_baseline(ne, seconds=3.0):
    """The MHD oracle as it stands (OpenMP on all host cores) on a bounded
    sample of the MHD leg's workload (the Alfven wave on ne^3 elements of
    degree 3), for both solvers: rhs evaluations over sampled elements for
    about `seconds` each."""
    import numpy as np
    import oracle
    from paper_2108_06476_gb300 import workloads as W
    oracle.build()
    N = 3
    n = (ne, ne, ne)
    nelem, P = ne ** 3, (N + 1) ** 3
    xi, _ = oracle.lgl(N)
    u = W.alfven_wave(N, n, xi, 0.0)
    du = np.zeros_like(u)
    out = {"cores": os.cpu_count() or 1, "kind": "oracle", "unit": UNIT}
    for key, vf, sf in (("weak_form_hll", "central", "hll"), ("ec_flux_differencing", "ec", "ec")):
        probe = np.arange(0, nelem, max(1, nelem // 64))[:64]
        t = time.perf_counter()
        oracle.mhd_rhs(N, n, W.box(3), u, elems=probe, out=du, vflux=vf, sflux=sf)
        per_elem = (time.perf_counter() - t) / len(probe)
        count = int(min(nelem, max(64, 0.3 * seconds / max(per_elem, 1e-9))))
        elems = np.sort(np.random.default_rng(3).choice(nelem, size=count, replace=False))
        reps, el = 0, 0.0
        t = time.perf_counter()
        while reps == 0 or (el < seconds and reps < 20):
            oracle.mhd_rhs(N, n, W.box(3), u, elems=elems, out=du, vflux=vf, sflux=sf)
            reps += 1
            el = time.perf_counter() - t
        out[key] = {"value": count * P * reps / el,
                    "sample": f"{reps} oracle rhs evaluation(s) over {count} of {nelem} "
                              f"elements, {el:.1f} s"}
    return out


def max_over_ranks(ms, dist, device="cuda"):
    """The slowest rank's time (the job's time); identity without a process
    group."""
    if dist is None:
        return ms
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(nodes_per_rank, stages, steps, world, ms):
    """Whole-job DOF-rhs-evaluations per second (weak scaling: every rank
    advances its own replica)."""
    return nodes_per_rank * stages * steps * world / (ms / 1e3)


def cpu_baseline(spec, xi, u):
    """The oracle's rhs on a bounded sample of the workload (about 10 s with
    all host cores: elements sampled, or the whole mesh repeated)."""
    import numpy as np
    import oracle
    oracle.build()
    d, N, ne = spec["d"], spec["N"], spec["ne"]
    n = (ne,) * d
    from paper_2108_06476_gb300 import workloads as W
    dom = W.box(d)
    nelem = ne ** d
    P = (N + 1) ** d
    du = np.zeros_like(u)
    probe = np.arange(0, nelem, max(1, nelem // 512))[:512]
    t = time.perf_counter()
    oracle.rhs(d, N, n, dom, u, elems=probe, out=du)
    per_elem = (time.perf_counter() - t) / len(probe)
    count = int(min(nelem, max(512, 10.0 / max(per_elem, 1e-9))))
    elems = np.sort(np.random.default_rng(2).choice(nelem, size=count, replace=False))
    reps, el = 0, 0.0
    t = time.perf_counter()
    while reps == 0 or (el < 10.0 and reps < 50):
        oracle.rhs(d, N, n, dom, u, elems=elems, out=du)
        reps += 1
        el = time.perf_counter() - t
    cores = os.cpu_count() or 1
    value = count * P * reps / el
    # one core, the paper's single-thread PID protocol (best of up to five
    # timed evaluations of a smaller sample)
    one = elems[: max(16, min(count, int(2.0 / max(per_elem * cores, 1e-9))))]
    best = None
    for _ in range(5):
        t = time.perf_counter()
        oracle.rhs(d, N, n, dom, u, elems=one, out=du, nthreads=1)
        dt = time.perf_counter() - t
        best = dt if best is None else min(best, dt)
        if dt > 3.0:
            break
    oracle.rhs(d, N, n, dom, u, elems=one[:1], out=du, nthreads=cores)  # restore the team
    single = {"value": len(one) * P / best, "pid_s": best / (len(one) * P),
              "sample": f"best of up to 5 single-thread oracle rhs evaluations over "
                        f"{len(one)} elements"}
    return {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
            "cpu_model": cpu_model(),
            "sample": f"{reps} oracle rhs evaluation(s) over {count} of {nelem} elements "
                      f"({count * P} nodes each), {el:.1f} s, OpenMP on all host cores",
            "single_core": single}


def run_ours(args, spec, world, rank, local):
    import numpy as np
    import torch
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    from paper_2108_06476_gb300 import Mesh, RK_A, RK_B, lgl_nodes, build as dgbuild
    dgbuild.build()
    d, N, ne = spec["d"], spec["N"], spec["ne"]
    n = (ne,) * d
    xi, _ = lgl_nodes(N)
    u_host = make_state(spec, xi, seed=rank)
    M = ne ** d * (N + 1) ** d
    peaks = measured_peaks()
    FP64_PEAK = peaks["fp64_tflops"]
    FP32_PEAK = peaks["fp32_tflops"]
    from paper_2108_06476_gb300 import measure_fp64_issue
    fp64_issue = measure_fp64_issue()
    mesh = Mesh(d, N, n, precision="fp64")
    u0 = torch.from_numpy(u_host).cuda()
    checks = []
    head_elems = _sample_elements(ne ** d, 400, seed=N)
    head_gpu = {}
    u = u0.clone()
    du = mesh.empty_rhs()
    stream = torch.cuda.current_stream()

    def barrier():
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()

    def run_steps(m, uu, dd, k):
        # device CFL step + five stages with the update fused into the volume
        # kernel, replayed as one CUDA graph per step
        for _ in range(k):
            m.step_cfl(uu, cfl=0.5, graph=True)

    def timed(fn):
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fn()
        e1.record(stream)
        barrier()
        return max_over_ranks(e0.elapsed_time(e1), dist)

    # ---- FP64: headline ----
    run_steps(mesh, u, du, args.warmup)
    with ClockSampler(local) as clk:
        ms = timed(lambda: run_steps(mesh, u, du, args.steps))
    mesh.check()
    value = job_value(M, 5, args.steps, world, ms)
    # the wave-speed pass (it also writes dt) and five stages of a face and a
    # volume kernel
    launches_per_step = 1 + 5 * 2

    # ---- kernel timings (dominant kernel: volume) ----
    def kernel_ms(m, uu, dd, part, reps=10):
        m.rhs_part(uu, dd, 1)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(reps):
            m.rhs_part(uu, dd, part)
        b.record(stream)
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps

    # rhs-only rate: 50 back-to-back dg_rhs calls (surface + volume kernels,
    # du written), the paper's PID without the stage updates
    u.copy_(u0)
    rhs_reps = 50
    mesh.rhs(u, du)
    ms_rhs = timed(lambda: [mesh.rhs(u, du) for _ in range(rhs_reps)])
    rhs_only = {"value": M * rhs_reps * world / (ms_rhs / 1e3), "unit": UNIT,
                "ms_per_rhs": ms_rhs / rhs_reps, "calls": rhs_reps}

    u.copy_(u0)
    head_gpu["fp64"] = mesh.rhs(u0).cpu().numpy().reshape(-1, d + 2, (N + 1) ** d)[head_elems]
    # the dominant kernel of the timed region is the fused volume kernel
    # (flux differencing, lifting and the stage update); parts=6 launches it
    # as in stages 2-5 (k read and written) with B = 0 (u unchanged)
    vol_ms = kernel_ms(mesh, u, du, 6)
    rhs_vol_ms = kernel_ms(mesh, u, du, 2)
    surf_ms = kernel_ms(mesh, u, du, 1)
    oc = counted_ops(args.workload) if args.elements == 0 else None
    flops_hand = volume_flops_per_node(d, N)
    flops_node = oc["volume_fused_per_node"] if oc else flops_hand
    flops_rhs_node = oc["volume_rhs_per_node"] if oc else flops_hand
    achieved = flops_node * M / (vol_ms / 1e3) / 1e12
    traffic = ncu_traffic(f"fp64_volume_{d}d_n{N}")
    # the hardware's view: FP64 flops the kernel executes per node (ncu
    # DADD + DMUL + 2 DFMA thread instructions), at the live kernel time
    counted_node = ncu_record(f"fp64_volume_{d}d_n{N}", "fp64_flops_executed_per_node")
    counted = None
    if counted_node is not None:
        c_ach = counted_node * M / (vol_ms / 1e3) / 1e12
        counted = {"flops_per_node": counted_node, "achieved": c_ach,
                   "frac": c_ach / FP64_PEAK}

    # ---- the memory-streaming kernels on the headline mesh ----
    # stand-alone stage update (dg_rk_stage: u, k and du read, k and u
    # written, 200 B per node; the step fuses it into the volume kernel) and
    # the compensated integrals (u read, 40 B per node; double-double sums
    # and two logarithms per node in FP64), against the measured copy
    # bandwidth
    streaming = None
    if not args.no_streaming:
        hbm = measured_hbm_gbs()
        u2 = u.clone()
        reps = 10
        mesh.rk_reset()  # k = 0: the timed updates stay tiny (dt 1e-9)
        mesh.rk_stage(u2, du, RK_A[1], RK_B[1], 1.0e-9)
        ms_rk = timed(lambda: [mesh.rk_stage(u2, du, RK_A[1], RK_B[1], 1.0e-9)
                               for _ in range(reps)]) / reps
        mesh.rk_reset()
        mesh.integrals(u2)
        ms_int = timed(lambda: [mesh.integrals(u2) for _ in range(3)]) / 3
        del u2
        b_rk, b_int = 5 * (d + 2) * 8 * M, (d + 2) * 8 * M
        streaming = {
            "hbm_peak_gbs": hbm, "hbm_peak_source": "MEASURED_PEAKS.json (copy, read + write)",
            "rk_stage": {"ms": ms_rk, "bytes": b_rk, "gbs": b_rk / ms_rk / 1e6,
                         "frac": None if hbm is None else b_rk / ms_rk / 1e6 / hbm},
            "integrals": {"ms": ms_int, "bytes": b_int, "gbs": b_int / ms_int / 1e6,
                          "frac": None if hbm is None else b_int / ms_int / 1e6 / hbm,
                          "note": "includes the host read of the 7 sums; FP64 arithmetic "
                                  "(two logs and seven double-double sums per node)"}}

    # ---- FP32 kernels with FP64 state and RK accumulation ----
    fp32 = None
    if not args.no_fp32:
        mesh32 = Mesh(d, N, n, precision="fp32")
        u32 = u0.clone()
        du32 = mesh32.empty_rhs()
        ref64 = mesh.rhs(u0).double()
        r32 = mesh32.rhs(u0, du32).double()
        err32 = float(torch.linalg.norm(r32 - ref64) / torch.linalg.norm(ref64))
        head_gpu["fp32"] = r32.cpu().numpy().reshape(-1, d + 2, (N + 1) ** d)[head_elems]
        del ref64, r32
        run_steps(mesh32, u32, du32, args.warmup)
        ms32 = timed(lambda: run_steps(mesh32, u32, du32, args.steps))
        mesh32.check()
        u32.copy_(u0)
        vol32 = kernel_ms(mesh32, u32, du32, 2)
        fp32 = {"value": M * 5 * args.steps * world / (ms32 / 1e3), "unit": UNIT,
                "ms_per_step": ms32 / args.steps, "speedup_vs_fp64": ms / ms32,
                "rhs_rel_l2_vs_fp64": err32,
                "volume_kernel_ms": vol32,
                "volume_tflops": flops_rhs_node * M / (vol32 / 1e3) / 1e12,
                "volume_frac_of_fp32_peak": flops_rhs_node * M / (vol32 / 1e3) / 1e12
                / FP32_PEAK}
        del mesh32, u32, du32

    # ---- end to end through the C ABI with a host buffer ----
    # dg_step_cfl_host per step: the state enters from pinned host memory
    # (read by the wave-speed pass) and leaves to it (stored by the last
    # stage), synchronously; all host-device bytes cross inside the region
    e2e = None
    if not args.no_e2e:
        uh = torch.empty(u0.numel(), dtype=torch.float64, pin_memory=True)
        uh.copy_(u0.cpu())

        def e2e_steps(k):
            for _ in range(k):
                mesh.step_cfl_host(uh, cfl=0.5, n_steps=1)

        e2e_steps(1)
        ms_e = timed(lambda: e2e_steps(args.steps))
        nbytes = u0.numel() * 8
        e2e = {"value": M * 5 * args.steps * world / (ms_e / 1e3), "unit": UNIT,
               "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes}

    # ---- batched ensemble: 48 members (seed 0), N in {3,4,5}, n in [8,24] ----
    ensemble = None
    if not args.no_ensemble:
        ensemble = run_ensemble(args, timed, rank, checks)

    # ---- VJP configuration ----
    vjp = None if args.no_vjp else run_vjp(args, timed)

    # ---- the other configured cases (rates only) ----
    configs = None
    if not args.no_configs:
        configs = run_configs(args, timed, checks)

    # ---- the paper's curvilinear benchmark setup ----
    curved = None
    if not args.no_curved:
        curved = run_curved(args, timed)

    # ---- 3D ideal MHD (Alfven wave) ----
    mhd = None
    if not args.no_mhd:
        mhd = run_mhd(args, timed, kernel_ms)

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "d": d, "N": N, "elements_per_dim": ne,
                   "nodes": M, "volume_flux": "ranocha", "surface_flux": "llf", "cfl": 0.5,
                   "parallelism": f"replicas{world}" if world > 1 else "single",
                   "l2": "inputs larger than L2 (state alone is "
                         f"{M * (d + 2) * 8 / 1e6:.0f} MB per buffer)"},
        "gpu_launches": launches_per_step * args.steps,
        "roofline": {"bound": "alu", "achieved": achieved, "peak": FP64_PEAK,
                     "unit": "TFLOP/s", "frac": achieved / FP64_PEAK,
                     "traffic": None if traffic is None else traffic * M,
                     "kernel": "volume_fx_kernel (FP64 mesh, stage update fused)",
                     "note": "the pair fluxes run on 64-bit integers, so the algorithmic "
                             "operations exceed the FP64 FMA rate: frac counts them against it, "
                             "counted.frac the FP64 instructions left",
                     "peak_source": f"measured: dg_measure_peaks FP64 FMA probe on "
                                    f"{peaks['sm_count']} SMs (cudaDeviceProp); nominal "
                                    f"{nominal_peaks(peaks['sm_count'])['fp64_tflops']:.3f} "
                                    f"TFLOP/s at {NOMINAL_SM_MHZ:.0f} MHz",
                     "fp32_peak_measured": FP32_PEAK,
                     "flops_per_node": flops_node,
                     "flops_source": ("oracle operation count (tests/golden/op_counts.json): "
                                      "primitives, d N/2 pair fluxes with their accumulation, "
                                      "lifting and the fused stage update; log, division, "
                                      "square root one each") if oc else "hand count",
                     "flops_per_node_hand_count_rhs": flops_hand,
                     "kernel_ms": vol_ms,
                     "counted": counted,
                     "fp64_issue_cycles": dict(fp64_issue, note=(
                         "SM cycles per dependent FP64 FMA, one warp per SM, 32 active lanes "
                         "and one (dg_measure_fp64_issue)"))},
        "kernels_ms": {"volume_fused_stage": vol_ms, "volume_rhs_only": rhs_vol_ms,
                       "surface": surf_ms},
        "rhs_only": rhs_only,
        "streaming_kernels": streaming,
        "fp32": fp32,
        "ensemble": ensemble,
        "vjp": vjp,
        "curved": curved,
        "mhd": mhd,
        "configs": configs,
        "e2e": e2e,
        "clocks": clk.summary(),
    }
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(spec, xi, u_host)
        line["cpu_baseline"]["configs"] = oracle_config_rates(0.5)
        oracle_checks(line, checks, (d, N, n, u_host, head_elems, head_gpu))
        if mhd is not None:
            mhd["cpu_baseline"] = mhd_cpu_baseline(args.mhd_elements)
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default=DEFAULT_WORKLOAD)
    ap.add_argument("--elements", type=int, default=0,
                    help="override elements per dimension (small cases for profiling)")
    ap.add_argument("--no-fp32", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-curved", action="store_true")
    ap.add_argument("--no-configs", action="store_true")
    ap.add_argument("--no-pid", action="store_true",
                    help="curved section: skip the 4^3 PID sweep")
    ap.add_argument("--curved-elements", type=int, default=64,
                    help="elements per direction of the curved throughput case")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-mhd", action="store_true")
    ap.add_argument("--mhd-elements", type=int, default=64,
                    help="MHD section: elements per dimension of the Alfven-wave mesh")
    ap.add_argument("--no-ensemble", action="store_true")
    ap.add_argument("--no-vjp", action="store_true")
    ap.add_argument("--no-streaming", action="store_true")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    spec = dict(WORKLOADS[args.workload])
    if args.elements > 0:
        spec["ne"] = args.elements
    world, rank, local = dist_setup()
    if args.impl == "reference":
        run_reference(args, spec, world, rank)
    else:
        run_ours(args, spec, world, rank, local)


if __name__ == "__main__":
    main()
