#!/usr/bin/env python3
"""Benchmark: gate-applications/s of a 30-qubit random brickwork circuit (depth 40, complex64) on one GB300.

One step = one full simulation of the circuit through libqsim: |0...0>, every pass of the planned circuit
(fused dense blocks on tensor cores or CUDA cores, diagonal passes), then the readouts the paper's
benchmarks use -- <Z_i>, <Z_i Z_{i+1}> and 1000 measurement samples (Sec. 2.2: 1000 shots per circuit).
value = unfused input gates x steps x ranks / max-over-ranks device time of the steps.

Also reported: the plain per-gate path and every fused variant (ms/step, passes, infidelity on the
20-qubit instance of the same generator against this library's complex128 per-gate path, which the test
suite pins to the FP64 oracle), the live per-pass roofline of the dominant
kernel, an end-to-end number through the public API with host buffers, SM clocks during the timed
region, and the FP64 oracle timed on the host cores on a bounded sample (cpu_baseline).

--impl reference times the oracle itself (the reference arm: there is no upstream code for this paper);
besides that arm, only the cpu_baseline legs execute the oracle.
Multi-GPU (--gpus N under torchrun): every rank simulates its own seeded instance (independent problems,
no data-path collective) -> weak scaling.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import re
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

UNIT = "gate-applications/s"
METRIC = "gate-applications/s, 30-qubit random brickwork depth 40 (Haar U(2) + CZ), complex64, 1000 shots"
SEED = 3


def parse_args():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=5)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--n", type=int, default=30)
    p.add_argument("--depth", type=int, default=40)
    p.add_argument("--shots", type=int, default=1000)
    p.add_argument("--path", default="auto", help="auto | " + " | ".join(PATHS))
    p.add_argument("--no-variants", action="store_true", help="skip the secondary path measurements")
    p.add_argument("--no-accuracy", action="store_true", help="skip the 20-qubit infidelity check")
    p.add_argument("--no-cpu", action="store_true", help="skip the cpu_baseline leg")
    p.add_argument("--no-configs", action="store_true",
                   help="skip the other configurations' runs after the headline line (N = 1 only)")
    p.add_argument("--configs-out", default=os.path.join("bench_out", "bench_configs.jsonl"),
                   help="file (relative to the repository root unless absolute) for the other configurations' "
                        "full JSON lines; a summary of each goes into the headline line")
    p.add_argument("--cpu-seconds", type=float, default=12.0)
    p.add_argument("--probe-seconds", type=float, default=1.5,
                   help="seconds per operand type of the tensor-core rate probe (0: skip it, no tensor fraction)")
    p.add_argument("--count", type=int, default=256, help="tfim_batch: number of circuits")
    p.add_argument("--nmax", type=int, default=24, help="tfim_batch: largest circuit width")
    p.add_argument("--workload", default="brickwork30",
                   choices=["brickwork30", "qft28", "tfim_batch", "pairs34", "brick14", "qpe33", "rcs33", "tfim33",
                            "spill33", "passes"],
                   help="brickwork30 (the headline line), qft28, tfim_batch (256 TFIM circuits), pairs34, "
                        "brick14 (14-qubit complex128, latency-bound)")
    return p.parse_args()


# ---- distributed plumbing (independent replicas; the only collectives are a barrier and a max) ---------------
def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def dist_init(ws):
    if ws <= 1:
        return None
    import torch.distributed as dist
    os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
    dist.init_process_group(backend="gloo")
    return dist


def barrier(dist):
    if dist is not None:
        dist.barrier()


def allmax(dist, x: float) -> float:
    if dist is None:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---- clocks during the timed region --------------------------------------------------------------------------
class Clocks:
    FIELDS = ("index,uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid):
        self.uuid = uuid
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(prefix="clocks.", suffix=".csv")
            os.close(fd)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 10:
                continue
            if self.uuid and parts[1] != self.uuid:
                continue
            rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None
        sm = [num(r[2]) for r in rows if num(r[2]) is not None]
        mx = [num(r[3]) for r in rows if num(r[3]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[6 + i].lower() == "active"})
        sm.sort()
        return {"sm_mhz": sm[len(sm) // 2] if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ---- roofline inputs -----------------------------------------------------------------------------------------
def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return d, "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}, "fallback"


KERNEL_SOURCES = {"dense_small": ["k_gates.cu"], "diag": ["k_gates.cu"], "dense_tile": ["k_gates.cu"],
                  "tc": ["k_tc.cu", "k_tc7.cu", "tc_ptx.cuh", "tmem_io.cuh"],
                  "tc_pair": ["k_tc_pair.cu", "tc_ptx.cuh", "tmem_io.cuh"]}


def source_sha(kind):
    """Hash of the code a kernel kind is built from, comments and layout removed (a profile's counters apply
    only while the code is unchanged)."""
    h = hashlib.sha256()
    for f in KERNEL_SOURCES[kind]:
        src = open(os.path.join(ROOT, "paper_2511_14664_gb300", "csrc", f)).read()
        src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
        src = re.sub(r"//[^\n]*", " ", src)
        h.update(" ".join(src.split()).encode())
    return h.hexdigest()[:12]


def profiled_traffic(kind, n):
    """DRAM bytes per launch from a committed ncu summary (profiles/*.md or *.txt lines 'bench-traffic: {...}'),
    used only while the kernel source is unchanged since the capture; scaled by 2^(n - n_captured)."""
    sha = source_sha(kind)
    pdir = os.path.join(ROOT, "profiles")
    if not os.path.isdir(pdir):
        return None
    for fn in sorted(os.listdir(pdir)):
        if not fn.endswith((".txt", ".md")):
            continue
        for line in open(os.path.join(pdir, fn)):
            m = re.match(r"\s*bench-traffic:\s*(\{.*\})\s*$", line)
            if not m:
                continue
            try:
                d = json.loads(m.group(1))
            except ValueError:
                continue
            if d.get("kind") == kind and d.get("source_sha") == sha:
                return float(d["bytes_per_launch"]) * 2.0 ** (n - int(d["n"]))
    return None


def tensor_rates(qsim, uuid, seconds):
    """Dense tensor-core rates of this GPU, measured live: an MMA-only tcgen05 loop on every SM in the form the
    block kernels issue (A in tensor memory, B in shared memory, M = N = 128, FP32 accumulation), `seconds`
    per operand type, SM clocks sampled meanwhile."""
    clocks = Clocks(uuid)
    clocks.start()
    out = {}
    for kind in ("tf32", "bf16", "fp16"):
        out[kind] = qsim.tc_peak(kind, 128, seconds)[0]
    clk = clocks.stop()
    out.update({"unit": "TFLOP/s", "sm_mhz": clk.get("sm_mhz"), "reasons": clk.get("reasons"),
                "how": f"tcgen05 MMA-only loop, one CTA per SM, A in TMEM, B in SMEM (SW128), M = N = 128, "
                       f"{seconds:g} s per type, CUDA events"})
    return out


PREC_RATE = {1: "tf32", 2: "bf16", 3: "bf16", 4: "fp16"}


# ---- the simulation step -------------------------------------------------------------------------------------
PATHS = {
    # name: (mode, max_fused, precision, tc_min_k)
    "plain": (0, 1, 0, 5),
    "simt4": (1, 4, 0, 5),
    "simt5": (1, 5, 0, 5),
    "tf32x3": (1, 6, 1, 5),
    "bf16x3": (1, 6, 2, 5),
    "bf16x6": (1, 6, 3, 5),
    "tf32x3_k5": (1, 5, 1, 5),
    "bf16x6_k5": (1, 5, 3, 5),
    "fp16x3": (1, 6, 4, 5),        # FP16 split products (3xTF32 where a block has the line-group / pair-rows path)
    "fp16x3_pairs": (1, 6, 4, 5, 1),  # the same, consecutive blocks paired into one pass
    "fp16x3_k7": (1, 7, 4, 5),     # FP16 split products with 7-qubit blocks (fewer passes)
}


def make_plan(qsim, circuit, path, use_graph=False):
    mode, k, prec, tcmin = PATHS[path][:4]
    pairs = len(PATHS[path]) > 4 and PATHS[path][4] == 1
    return qsim.Plan(circuit, qsim.C64, mode=mode, max_fused=k, precision=prec, tc_min_k=tcmin, use_graph=use_graph,
                     pair_blocks=pairs)


def count_readout_launches(n):
    """Kernels of one expect_z_and_sample call: <Z> statistics (one kernel below 12 qubits; else warp
    segments, their final sum, high-bit partials, their final sum), then uniforms, segment sums (left by the
    <Z> pass from 12 qubits on), chunk sums, scan, sample."""
    return 1 + 5 if n < 12 else 4 + 4


def count_step_launches(plan, n):
    """Kernels one bench step launches: the basis set-up (unless the first block generates it), every pass's
    kernels, the readout."""
    return (0 if generates_input(plan) else 1) + sum(q["launches"] for q in plan.pass_list) + count_readout_launches(n)


def generates_input(plan):
    """True when the plan's first pass is a 3xTF32 / BF16x3 tensor-core block, which execute_from_basis runs
    on a generated basis state (its algorithmic bytes are then the writes alone)."""
    q = plan.pass_list[0] if plan.pass_list else None
    return bool(q) and q["kind"] in ("tc", "tc_pair") and q["precision"] != 3


def timed_steps(qsim, torch, st, plan, steps, shots, per_pass=True):
    """Run `steps` steps; returns (total_ms, per-pass ms list summed over steps). With per_pass, CUDA events
    time the passes: around every pass, or, when every pass is of one kind, around the run of passes as a
    whole (an event between two block kernels would stop the second from overlapping the first one's tail
    as a programmatic dependent launch); the run's time is then shared equally among its passes."""
    stream = torch.cuda.current_stream()
    npass = len(plan.pass_list)
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    pass_ms = [0.0] * npass
    uniform = len({q["kind"] for q in plan.pass_list}) == 1
    nev = 2 if uniform else npass + 1
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(nev)] for _ in range(steps)] if per_pass else None
    gen = generates_input(plan)
    torch.cuda.synchronize()
    t0.record(stream)
    for s in range(steps):
        # |0>, then the plan: a first tensor-core block generates |0> itself instead of reading a set-up state
        if per_pass:
            ev = evs[s]
            if not gen:
                st.set_basis(0)
            ev[0].record(stream)
            if uniform:
                plan.execute_from_basis(st, 0)
                ev[1].record(stream)
            else:
                plan.execute_from_basis(st, 0, 1)
                ev[1].record(stream)
                for i in range(1, npass):
                    plan.execute_range(st, i, 1)
                    ev[i + 1].record(stream)
        else:
            plan.execute_from_basis(st, 0)
        st.expect_z_and_sample(1000 + s, shots)   # <Z_i>, <Z_i Z_i+1> and the shots, one read of the state
    t1.record(stream)
    torch.cuda.synchronize()
    if per_pass:
        for ev in evs:
            if uniform:
                share = ev[0].elapsed_time(ev[1]) / npass
                for i in range(npass):
                    pass_ms[i] += share
            else:
                for i in range(npass):
                    pass_ms[i] += ev[i].elapsed_time(ev[i + 1])
    return t0.elapsed_time(t1), pass_ms


def path_states_at(qsim, W, n_small, depth, paths):
    """Final complex64 states of every path on the n_small-qubit instance of the same generator (accuracy is
    measured on this instance: the full-size state has no FP64 reference)."""
    c = W.brickwork(n_small, depth, seed=SEED)
    out = {}
    st = qsim.State(n_small, qsim.C64)
    for path in paths:
        plan = make_plan(qsim, c, path)
        st.set_basis(0)
        plan.execute(st)
        out[path] = st.get_state().astype("complex128")
        plan.close()
    st.close()
    return c, out


def accuracy_vs(ref, states, label):
    """Per path: normalised infidelity 1 - |<ref|psi>|^2 / (<ref|ref><psi|psi>), max amplitude error and norm
    deviation against `ref`."""
    import numpy as np
    acc = {}
    nr = float(np.vdot(ref, ref).real)
    for name, psi in states.items():
        npsi = float(np.vdot(psi, psi).real)
        inf = max(0.0, 1.0 - abs(np.vdot(ref, psi)) ** 2 / (nr * npsi))
        acc[name] = {"n": int(round(math.log2(len(ref)))), "infidelity": inf,
                     "max_amp_err": float(np.max(np.abs(psi - ref))), "norm_dev": abs(npsi - 1.0), "reference": label}
    return acc


def gpu_c128_reference(qsim, c):
    """The library's complex128 per-gate path on the same circuit (used only when the oracle leg is off)."""
    rp = qsim.Plan(c, qsim.C128, mode=0, max_fused=1)
    rs = qsim.State(c.n, qsim.C128)
    rs.set_basis(0)
    rp.execute(rs)
    ref = rs.get_state()
    rp.close()
    rs.close()
    return ref


def oracle_reference(oracle_mod, c):
    """cpu_baseline leg: the FP64 oracle's final state of the accuracy instance, and the seconds it took."""
    t = time.perf_counter()
    ref = oracle_mod.run(c)
    return ref, time.perf_counter() - t


def cpu_baseline(oracle_mod, W, n_full, depth, seconds):
    """The FP64 oracle on the host cores: the first gates of the 25-qubit instance of the same generator,
    run until `seconds` elapse; gate-applications/s scaled by 2^(n_s - n_full) (work per gate ~ 2^n)."""
    n_s = min(25, n_full)
    c = W.brickwork(n_s, depth, seed=SEED)
    psi = oracle_mod.basis(n_s, 0)
    t = time.perf_counter()
    g = 0
    for gate in c.gates:
        oracle_mod.apply_gate(psi, n_s, gate.targets, gate.controls, gate.matrix)
        g += 1
        if time.perf_counter() - t > seconds:
            break
    dt = time.perf_counter() - t
    rate = g / dt * 2.0 ** (n_s - n_full)
    return {"value": rate, "unit": UNIT, "cores": oracle_mod.num_threads(), "kind": "oracle",
            "sample": f"first {g} gates of the {n_s}-qubit instance of the generator in {dt:.1f} s, "
                      f"rate scaled by 2^({n_s}-{n_full}) (work per gate ~ 2^n)"}


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    import oracle as oracle_mod
    import workloads as W
    n_s = min(24, args.n)
    c = W.brickwork(n_s, args.depth, seed=SEED)
    per_step_gates = 24
    psi = oracle_mod.basis(n_s, 0)
    gi = 0

    def step():
        nonlocal gi
        for _ in range(per_step_gates):
            g = c.gates[gi % len(c.gates)]
            oracle_mod.apply_gate(psi, n_s, g.targets, g.controls, g.matrix)
            gi += 1
    for _ in range(args.warmup):
        step()
    t = time.perf_counter()
    for _ in range(args.steps):
        step()
    dt = time.perf_counter() - t
    rate = per_step_gates * args.steps / dt * 2.0 ** (n_s - args.n)
    sample = (f"each step: {per_step_gates} gates of the {n_s}-qubit instance of the generator on the FP64 "
              f"oracle, rate scaled by 2^({n_s}-{args.n})")
    line = {"impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * dt / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"random brickwork n={args.n} depth={args.depth} seed={SEED}",
                       "global_batch": 1, "seq_len": None, "parallelism": "replicas"},
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": oracle_mod.num_threads(), "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def run_ours(args):
    ws, rank, local = dist_env()
    dist = dist_init(ws)
    import numpy as np
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim

    torch.cuda.set_device(local)
    qsim.lib()
    dev = torch.cuda.current_device()
    uuid = None
    try:
        uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    n, depth, shots = args.n, args.depth, args.shots
    circuit = W.brickwork(n, depth, seed=SEED + rank)
    G = len(circuit)
    st = qsim.State(n, qsim.C64)

    # candidate paths (tensor-core variants only where the library supports them)
    cands = ["fp16x3_k7", "fp16x3", "tf32x3", "fp16x3_pairs", "bf16x3", "bf16x6", "tf32x3_k5", "bf16x6_k5", "simt4", "simt5"]
    plans = {}
    for name in cands + ["plain"]:
        try:
            plans[name] = make_plan(qsim, circuit, name)
            plans[name].pass_list = plans[name].passes()
        except qsim.QsimError:
            pass
    # accuracy of each path on the 20-qubit instance (equal-accuracy comparison), against the FP64 oracle
    # (the cpu_baseline leg, rank 0 at N = 1) or else the library's complex128 per-gate path
    acc, oracle_acc_s = {}, None
    if rank == 0 and not args.no_accuracy:
        c_small, states = path_states_at(qsim, W, min(20, n), depth, list(plans))
        if ws == 1 and not args.no_cpu:
            import oracle as oracle_mod
            ref, oracle_acc_s = oracle_reference(oracle_mod, c_small)
            acc = accuracy_vs(ref, states, "FP64 oracle")
        else:
            acc = accuracy_vs(gpu_c128_reference(qsim, c_small), states, "complex128 per-gate path of this library")

    def quick(name, steps=1, warm=1):
        p = plans[name]
        timed_steps(qsim, torch, st, p, warm, shots, per_pass=False)
        ms, _ = timed_steps(qsim, torch, st, p, steps, shots, per_pass=False)
        return ms / steps

    variants = {}
    if not args.no_variants:
        for name in plans:
            if name == "plain":
                continue
            variants[name] = {"ms_per_step": quick(name), "passes": len(plans[name].pass_list)}
    if args.path == "auto":
        # equal accuracy: infidelity on the 20-qubit instance at least 10x inside the 1e-9 bar, since the
        # 30-qubit state itself is not checked element by element
        ok = [k for k in variants if (not acc or acc[k]["infidelity"] <= 1e-10)]
        main = min(ok, key=lambda k: variants[k]["ms_per_step"]) if ok else ("tf32x3" if "tf32x3" in plans else "simt4")
    else:
        main = args.path
    plan = plans[main]

    rates = tensor_rates(qsim, uuid, args.probe_seconds if args.steps >= 3 else min(args.probe_seconds, 0.5)) \
        if args.probe_seconds > 0 else None

    # ---- the timed region -------------------------------------------------------------------------------
    timed_steps(qsim, torch, st, plan, args.warmup, shots, per_pass=True)
    clocks = Clocks(uuid)
    barrier(dist)
    torch.cuda.synchronize()
    clocks.start()
    total_ms, pass_ms = timed_steps(qsim, torch, st, plan, args.steps, shots, per_pass=True)
    torch.cuda.synchronize()
    clk = clocks.stop()
    barrier(dist)
    t_max = allmax(dist, total_ms)
    value = G * args.steps * ws / (t_max / 1000.0)

    # ---- roofline of the dominant pass kind ------------------------------------------------------------------
    peaks, peak_src = measured_peaks()
    by_kind = {}
    gen = generates_input(plan)
    for i, (info, ms) in enumerate(zip(plan.pass_list, pass_ms)):
        d = by_kind.setdefault(info["kind"], {"ms": 0.0, "bytes": 0.0, "launches": 0, "flops": 0.0, "floor_s": 0.0})
        d["ms"] += ms
        d["bytes"] += info["algorithmic_bytes"] * (0.5 if (i == 0 and gen) else 1.0) * args.steps
        d["launches"] += args.steps
        if info["kind"] in ("tc", "tc_pair"):
            mult = {1: 3, 2: 3, 3: 6, 4: 3}[info["precision"]]
            blocks = 2 if info["kind"] == "tc_pair" else 1
            # real GEMM per amplitude: 2 * (2 * 2^k) MACs per complex output -> 8 * 2^k flops x split products
            f = (2.0 ** n) * 8 * (2 ** info["k"]) * mult * blocks * args.steps
            d["flops"] += f
            if rates is not None:  # the time these flops take at the measured rate of this block's operand type
                d["floor_s"] += f / (rates[PREC_RATE[info["precision"]]] * 1e12)
    dom = max(by_kind, key=lambda k: by_kind[k]["ms"])
    dk = by_kind[dom]
    avg_s = dk["ms"] / dk["launches"] / 1000.0
    bytes_per_launch = dk["bytes"] / dk["launches"]
    gbs = bytes_per_launch / avg_s / 1e9
    hbm_frac = gbs / peaks["hbm_gbs"]
    roof = {"bound": "hbm", "achieved": gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s", "frac": hbm_frac,
            "traffic": profiled_traffic(dom, n), "kernel": dom, "launches_per_step": dk["launches"] // args.steps,
            "avg_launch_ms": avg_s * 1000.0, "share_of_step": dk["ms"] / total_ms, "peak_source": peak_src}
    if dom in ("tc", "tc_pair") and dk["flops"] > 0 and rates is not None:
        tflops = dk["flops"] / dk["launches"] / avg_s / 1e12
        # the rate of each block's operand type, measured on this GPU in this run (tensor_rates); a plan that
        # mixes types gets the rate that takes the same time for the same flops
        used = sorted({PREC_RATE[p["precision"]] for p in plan.pass_list if p["kind"] == dom})
        tpeak = dk["flops"] / dk["floor_s"] / 1e12
        roof["tensor"] = {"achieved": tflops, "peak": tpeak, "unit": "TFLOP/s", "frac": tflops / tpeak,
                          "peak_source": f"measured: {' + '.join(used)} MMA-only loop on this GPU, this run"
                                         + (" (flop-weighted over the blocks' types)" if len(used) > 1 else "")}
        if tflops / tpeak > hbm_frac:
            roof = {**roof, "bound": "tensor", "achieved": tflops, "peak": tpeak, "unit": "TFLOP/s",
                    "frac": tflops / tpeak}

    # ---- plain per-gate path (the baseline the fused forms must beat) -------------------------------------------
    plain = None
    if not args.no_variants and "plain" in plans:
        pp = plans["plain"]
        timed_steps(qsim, torch, st, pp, 1, shots, per_pass=False)
        ms, _ = timed_steps(qsim, torch, st, pp, 1, shots, per_pass=False)   # groups of gates share a pass
        by_pass_ms, pms = timed_steps(qsim, torch, st, pp, 1, shots, per_pass=True)  # one pass a gate
        dense = [(i, m) for i, (i2, m) in enumerate(zip(pp.pass_list, pms)) if pp.pass_list[i]["kind"] == "dense_small"]
        dense_bytes = sum(pp.pass_list[i]["algorithmic_bytes"] for i, _ in dense)
        dense_ms = sum(m for _, m in dense)
        plain = {"gates_per_s": G / (ms / 1000.0), "ms_per_step": ms, "passes": len(pp.pass_list),
                 "ms_per_step_gate_by_gate": by_pass_ms,
                 "per_gate_pass_gbs": dense_bytes / (dense_ms / 1000.0) / 1e9 if dense_ms > 0 else None}

    # ---- end to end through the public API with host buffers -----------------------------------------------------
    import ctypes
    h2d = sum(16 * (1 << (2 * len(g.targets))) + ctypes.sizeof(qsim.Gate) for g in circuit.gates)
    d2h = 8 * (2 * n - 1) + 8 * shots
    e2e_steps = max(1, min(args.steps, 3))
    torch.cuda.synchronize()
    t = time.perf_counter()
    for s in range(e2e_steps):
        qsim.plan_cache_clear()              # cold planning every step (no grouping reused across steps)
        p = make_plan(qsim, circuit, main)   # host gate list -> device (planning, upload, FP64 composition)
        p.execute_from_basis(st, 0)
        zi, zz, smp = st.expect_z_and_sample(5000 + s, shots)     # device -> host
        p.close()
    torch.cuda.synchronize()
    e2e_s = (time.perf_counter() - t) / e2e_steps
    e2e_val = allmax(dist, e2e_s)
    e2e = {"value": G * ws / e2e_val, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h}

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": t_max / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32" if main in ("plain", "simt4", "simt5") else main[:4],
        "precision": main,
        "data": "synthetic",
        "config": {"workload": f"random brickwork n={n} depth={depth} seed={SEED}(+rank), {G} gates, complex64",
                   "path": main, "passes": len(plan.pass_list), "global_batch": ws, "seq_len": None,
                   "parallelism": f"replicas x{ws}", "shots": shots,
                   "l2": f"state {2 ** n * 8 / 2 ** 30:.0f} GiB > L2 129 MB: inputs larger than L2, no flush"},
        "gpu_launches": args.steps * count_step_launches(plan, n),
        "roofline": roof,
        "clocks": clk,
        "e2e": e2e,
        "plain": plain,
        "variants": variants,
        "accuracy": acc,
        "plan_ms": plan.info["host_plan_ms"],
        "tensor_rates": rates,
    }
    if rank == 0 and ws == 1 and not args.no_cpu:
        import oracle as oracle_mod
        line["cpu_baseline"] = cpu_baseline(oracle_mod, W, n, depth, args.cpu_seconds)
        if oracle_acc_s is not None:
            line["cpu_baseline"]["accuracy_reference"] = (
                f"FP64 oracle on the {min(20, n)}-qubit instance of the generator ({oracle_acc_s:.1f} s on "
                f"{oracle_mod.num_threads()} cores); every path's accuracy line is measured against it")
    if rank == 0 and ws == 1 and not args.no_configs:
        # the other configurations, each in a process of its own after this one's timed region: full lines
        # to the --configs-out file, a summary of each in this line
        del st, plans, plan
        torch.cuda.empty_cache()
        line["configs"] = run_other_configs(args.configs_out)
    if rank == 0:
        print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()
    return 0


OTHER_CONFIGS = [
    # (workload, extra arguments): bounded runs of the other configurations of the benchmark set
    ("brick14", ["--steps", "10", "--warmup", "3"]),
    ("qft28", ["--steps", "3", "--warmup", "1"]),
    ("tfim_batch", ["--steps", "5", "--warmup", "2", "--no-variants", "--cpu-seconds", "3"]),
    ("pairs34", ["--steps", "1", "--warmup", "1", "--no-variants"]),
]


def run_other_configs(out_path):
    out_path = out_path if os.path.isabs(out_path) else os.path.join(ROOT, out_path)
    os.makedirs(os.path.dirname(out_path), exist_ok=True)
    summary = {}
    with open(out_path, "w") as f:
        for wl, extra in OTHER_CONFIGS:
            cmd = [sys.executable, os.path.join(ROOT, "bench.py"), "--workload", wl, *extra]
            t = time.perf_counter()
            try:
                r = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
                lines = [x for x in r.stdout.splitlines() if x.startswith("{")]
                rec = json.loads(lines[-1]) if (r.returncode == 0 and lines) else None
                err = None if rec else (r.stderr.strip().splitlines() or ["no output"])[-1][:300]
            except Exception as e:  # a failed secondary run must not take the headline line with it
                rec, err = None, f"{type(e).__name__}: {e}"[:300]
            wall = time.perf_counter() - t
            if rec is None:
                summary[wl] = {"error": err, "wall_s": wall}
                continue
            f.write(json.dumps(rec) + "\n")
            summary[wl] = {k: rec.get(k) for k in ("metric", "value", "unit", "ms_per_step", "dtype")}
            summary[wl]["path"] = rec.get("config", {}).get("path")
            summary[wl]["wall_s"] = wall
            for k in ("roofline", "accuracy_vs_oracle", "e2e"):
                if k in rec:
                    summary[wl][k] = rec[k]
    return summary


# ---- secondary workloads (their own JSON lines; the default run prints only the headline line) -----------------
def _common_line(metric, value, unit, args, ms, dtype, config, **extra):
    line = {"metric": metric, "value": value, "unit": unit, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": dtype,
            "data": "synthetic", "config": config}
    line.update(extra)
    return line


def _event_time(torch, fn, steps):
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(st)
    for i in range(steps):
        fn(i)
    e1.record(st)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / steps


def run_brick14(args):
    """14-qubit random brickwork (20 layers: Haar U(2) on every qubit + CZ on alternating pairs, 410 gates),
    complex128, full output vector. The state is 256 KiB, so every pass is L2-resident and the run is
    launch-, latency- and FP64-bound: plans of CUDA-core passes run in one resident cooperative launch (grid
    barriers between groups of gates or between passes), and the same plans launched pass by pass from CUDA
    graphs are timed beside them. Every path's final vector is compared with the per-gate path's (both complex128 on the GPU;
    the test suite pins the per-gate path to the FP64 oracle)."""
    import numpy as np
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    n, depth = 14, 20
    c = W.brickwork(n, depth, seed=1)
    st = qsim.State(n, qsim.C128)
    out = {}
    ref = None
    finals = {}
    for name, kw in [("plain", dict(mode=0, max_fused=1)), ("simt2", dict(mode=1, max_fused=2)),
                     ("simt3", dict(mode=1, max_fused=3)), ("simt4", dict(mode=1, max_fused=4)),
                     ("simt5", dict(mode=1, max_fused=5)),
                     ("simt3_per_pass", dict(mode=1, max_fused=3, launch_per_pass=True)),
                     ("simt4_per_pass", dict(mode=1, max_fused=4, launch_per_pass=True))]:
        p = qsim.Plan(c, qsim.C128, use_graph=True, **kw)

        def step(i, p=p):
            p.execute_from_basis(st, 0)
        for _ in range(max(3, args.warmup)):
            step(0)
        steps = max(10, args.steps)
        ms = _event_time(torch, step, steps)
        psi = st.get_state()
        finals[name] = psi
        if ref is None:
            ref = psi
        # FP64 arithmetic of the dense passes: every amplitude of a touched group is a 2^k-term complex dot
        # product (8 2^k real flops); diagonal and phase passes add a few flops per amplitude (not counted). A
        # resident plan may apply the gates themselves, or products of a few, which are fewer: counted gate by gate that
        # is an effective rate, which says nothing about the units and is not set against their peak.
        resident = bool(p.info["resident"])
        if resident:
            fp64 = sum(8.0 * (1 << len(g.targets)) * 2.0 ** (n - len(g.controls)) for g in c.gates
                       if np.count_nonzero(g.matrix - np.diag(np.diag(g.matrix))))
        else:
            fp64 = sum(8.0 * (1 << q["k"]) * 2.0 ** (n - q["nc"]) for q in p.passes()
                       if q["kind"] in ("dense_small", "dense_tile"))
        out[name] = {"ms_per_step": ms, "gates_per_s": len(c) / (ms / 1000.0), "passes": p.info["passes"],
                     "resident": resident, "fp64_gflop": None if resident else fp64 / 1e9,
                     "fp64_tflops": None if resident else fp64 / (ms / 1000.0) / 1e12,
                     "fp64_tflops_gate_by_gate": fp64 / (ms / 1000.0) / 1e12 if resident else None,
                     "us_per_pass": 1000.0 * ms / p.info["passes"],
                     "algorithmic_gb": p.info["algorithmic_bytes"] / 1e9,
                     "achieved_gbs": p.info["algorithmic_bytes"] / (ms / 1000.0) / 1e9,
                     "max_abs_diff_vs_plain": float(np.max(np.abs(psi - ref)))}
    best = min(out, key=lambda k: out[k]["ms_per_step"])
    kw = dict(mode=0, max_fused=1) if best == "plain" else dict(mode=1, max_fused=int(best[4]))
    if best.endswith("_per_pass"):
        kw["launch_per_pass"] = True
    # end to end through the public API: plan + execute + destroy (qsim_run) and the full vector to the host
    ts = []
    for i in range(max(3, args.warmup) + max(10, args.steps)):
        torch.cuda.synchronize()
        qsim.plan_cache_clear()  # cold planning in every timed run
        t = time.perf_counter()
        st.set_basis(0)
        st.run(c, **kw)
        v = st.get_state()
        ts.append(time.perf_counter() - t)
    e2e_s = float(np.median(ts[max(3, args.warmup):]))
    b = out[best]
    fp64_peak = qsim.fp64_peak(1.0)[0]
    line = _common_line("gate-applications/s, 14-qubit random brickwork (20 layers), complex128, full output vector",
                        b["gates_per_s"], UNIT, args, b["ms_per_step"], "f64",
                        {"workload": f"random brickwork n={n} depth={depth} seed=1, {len(c)} gates, complex128",
                         "path": best, "resident": b["resident"], "graph": not b["resident"],
                         "l2": "state 256 KiB: L2-resident by design (latency-bound configuration)"},
                        paths=out, gpu_launches=1 + (1 if b["resident"] else b["passes"]),
                        roofline={"bound": "alu", "achieved": b["fp64_tflops"], "peak": fp64_peak, "unit": "TFLOP/s",
                                  "frac": None if b["resident"] else b["fp64_tflops"] / fp64_peak, "traffic": None,
                                  "gate_by_gate": b["fp64_tflops_gate_by_gate"],
                                  "peak_source": "measured: independent FP64 FMA chains on every SM, this run",
                                  "note": "L2-resident state (no HBM traffic to speak of): FP64 arithmetic, barriers and "
                                          "latency. A resident plan runs products of gates, less arithmetic than the "
                                          "gates: gate_by_gate is an effective rate, not a share of the peak",
                                  "hbm_equivalent_gbs": b["achieved_gbs"]},
                        e2e={"value": len(c) / e2e_s, "unit": UNIT,
                             "h2d_bytes_per_step": int(sum(g.matrix.size * 16 + 8 * (len(g.targets) + len(g.controls)) for g in c.gates)),
                             "d2h_bytes_per_step": int(v.nbytes)})
    line["steps"] = max(10, args.steps)
    line["warmup"] = max(3, args.warmup)
    if not args.no_cpu:
        # cpu_baseline leg: the FP64 oracle on the same circuit (timed), and every path's final vector against it
        import oracle as oracle_mod
        t = time.perf_counter()
        ref = oracle_mod.run(c)
        dt = time.perf_counter() - t
        line["cpu_baseline"] = {"value": len(c) / dt, "unit": UNIT, "cores": oracle_mod.num_threads(),
                                "kind": "oracle", "sample": f"the whole {len(c)}-gate circuit once ({dt * 1e3:.1f} ms)"}
        acc = {}
        for name, psi in finals.items():
            ov = np.vdot(ref, psi)
            acc[name] = {"max_abs_err": float(np.max(np.abs(psi - ref))),
                         "infidelity": max(0.0, 1.0 - abs(ov) ** 2 / (np.vdot(ref, ref).real * np.vdot(psi, psi).real))}
        line["accuracy_vs_oracle"] = acc
    print(json.dumps(line))
    return 0


def run_qft(args):
    """28-qubit QFT of a seeded basis state: plain per-gate vs fused (k = 5), checked against the closed form
    on sampled amplitudes (|QFT x>_y = 2^{-n/2} exp(2 pi i x y / 2^n))."""
    import numpy as np
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    n = args.n if args.n != 30 else 28
    x = W.basis_index(n, 2)
    c = W.qft(n)
    st = qsim.State(n, qsim.C64)
    peaks, _ = measured_peaks()
    out = {}
    for name, kw in [("plain", dict(mode=0, max_fused=1)), ("simt5", dict(mode=1, max_fused=5)),
                     ("tf32x3_k5", dict(mode=1, max_fused=5, precision=1, tc_min_k=5)),
                     ("bf16x6_k5", dict(mode=1, max_fused=5, precision=3, tc_min_k=5)),
                     ("tf32x3_k6", dict(mode=1, max_fused=6, precision=1, tc_min_k=5)),
                     ("bf16x6_k6", dict(mode=1, max_fused=6, precision=3, tc_min_k=5)),
                     ("fp16x3_k6", dict(mode=1, max_fused=6, precision=4, tc_min_k=5)),
                     ("fp16x3_k7", dict(mode=1, max_fused=7, precision=4, tc_min_k=5))]:
        p = qsim.Plan(c, **kw)

        def step(i, p=p):
            st.set_basis(x)
            p.execute(st)
        for _ in range(max(1, args.warmup)):
            step(0)
        ms = _event_time(torch, step, max(1, args.steps))
        rng = np.random.default_rng(1)
        ys = np.sort(rng.choice(1 << n, size=4096, replace=False))
        got = st.tensor[torch.from_numpy(ys).cuda()].cpu().numpy().astype(np.complex128)
        ph = (np.uint64(x) * ys.astype(np.uint64)) & np.uint64((1 << n) - 1)
        ref = np.exp(2j * math.pi * ph.astype(np.float64) / (1 << n)) / math.sqrt(1 << n)
        out[name] = {"ms_per_step": ms, "gates_per_s": len(c) / (ms / 1000.0), "passes": p.info["passes"],
                     "algorithmic_gb": p.info["algorithmic_bytes"] / 1e9,
                     "achieved_gbs": p.info["algorithmic_bytes"] / (ms / 1000.0) / 1e9,
                     "max_err_sampled": float(np.max(np.abs(got - ref)))}
    best = min((k for k in out if k != "plain"), key=lambda k: out[k]["ms_per_step"])
    line = _common_line(f"gate-applications/s, {n}-qubit QFT (with swaps), complex64, fused (k = 5, 6) vs plain",
                        out[best]["gates_per_s"], UNIT, args, out[best]["ms_per_step"],
                        "f32" if best.startswith(("plain", "simt")) else best[:4],
                        {"workload": f"QFT n={n} from |x>, x={x}, {len(c)} gates", "path": best},
                        paths=out, peak_hbm_gbs=peaks["hbm_gbs"])
    print(json.dumps(line))
    return 0


def run_tfim_batch(args):
    """256 Trotterised TFIM chains (widths U{10..24}, steps U{8..32}, theta, phi ~ U(0, pi); seed 4) in one
    enqueue replayed from a CUDA graph: the persistent launch (fusion width tuned per circuit width) for the
    circuits below 20 qubits, tensor-core plans for the wider ones (3xTF32 with 6-qubit blocks or FP16X3 with
    up to 7, the faster reported); per-circuit <Z_i> and <Z_i Z_{i+1}>."""
    import numpy as np
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    batch = W.tfim_batch(args.count, seed=4, nmax=args.nmax)
    cs = [c for c, _, _ in batch]
    gates = sum(len(c) for c in cs)
    t = time.perf_counter()
    chosen = qsim.batch_autotune(cs)
    tune_s = time.perf_counter() - t
    # circuits of >= 20 qubits as tensor-core plans (3xTF32 with 6-qubit blocks, or FP16X3 with up to 7: the
    # faster is reported), the rest in the persistent launch
    tc_min_n = 20
    wide_paths = {}
    for prec in (1, 4):
        bb = qsim.Batch(cs, max_fused=0, precision=prec, tc_min_n=tc_min_n)
        for _ in range(max(1, args.warmup)):
            bb.execute(use_graph=True)
        wide_paths[prec] = (_event_time(torch, lambda i: bb.execute(use_graph=True), max(1, args.steps)), bb)
    tc_prec = min(wide_paths, key=lambda p: wide_paths[p][0])
    ms, b = wide_paths[tc_prec]
    wide_ms = {("tf32x3 k = 6" if p == 1 else "fp16x3 k <= 7"): round(v[0], 3) for p, v in wide_paths.items()}
    wide_paths[4 if tc_prec == 1 else 1][1].close()
    res = b.results()
    # the same batch in the states' own precision (persistent launch, wide circuits as own-precision plans)
    simt_only = None
    if not args.no_variants:
        bs = qsim.Batch(cs, max_fused=0)
        bs.execute(use_graph=True)
        ms_s = _event_time(torch, lambda i: bs.execute(use_graph=True), max(1, args.steps))
        rs = bs.results()
        simt_only = {"ms": ms_s, "gates_per_s": gates / (ms_s / 1000.0),
                     "max_abs_diff_zi_vs_main": max(float(np.max(np.abs(rs[i][0] - res[i][0]))) for i in range(len(cs)))}
        bs.close()
    # end to end: the one-shot call from host circuits to host results (qsim_batch_run: the GPU runs the
    # circuits already planned while the host plans the others), best of three; beside it the same batch
    # planned, then executed, with its breakdown
    e2e_runs = []
    for _ in range(3):
        torch.cuda.synchronize()
        qsim.plan_cache_clear()  # cold: only groupings repeated within this batch are reused
        t = time.perf_counter()
        _, rinfo = qsim.batch_run(cs, max_fused=0, precision=tc_prec, tc_min_n=tc_min_n)
        e2e_runs.append({"total_s": time.perf_counter() - t, "c_plan_and_enqueue_ms": rinfo["host_plan_ms"]})
    staged = []
    for _ in range(3):
        torch.cuda.synchronize()
        qsim.plan_cache_clear()
        t = time.perf_counter()
        b2 = qsim.Batch(cs, max_fused=0, precision=tc_prec, tc_min_n=tc_min_n)
        t_plan = time.perf_counter()
        b2.execute()
        b2.results()
        t_run = time.perf_counter()
        b2.close()
        staged.append({"total_s": time.perf_counter() - t, "plan_s": t_plan - t,
                       "c_plan_ms": b2.info["host_plan_ms"], "execute_results_s": t_run - t_plan})
    best = min(e2e_runs, key=lambda r: r["total_s"])
    e2e_s = best["total_s"]
    peaks, src = measured_peaks()
    gbs = b.info["algorithmic_bytes"] / (ms / 1000.0) / 1e9
    widths = sorted(set(c.n for c in cs))
    kmap = {str(n): chosen[[c.n for c in cs].index(n)] for n in widths}
    # Baselines the batched launch must beat: the same circuits one after another, each through its own
    # plan (CUDA-graph replay) and its own <Z_i>, <Z_i Z_i+1> readout: plain per-gate passes, and the fused
    # plans with the width the tuner chose.
    one_by_one = {}
    if not args.no_variants:
        states = {n: qsim.State(n, qsim.C64) for n in widths}
        for name, mk in (("plain", lambda c: dict(mode=qsim.RUN_PLAIN, max_fused=1)),
                         ("fused", lambda c: dict(mode=qsim.RUN_FUSED, max_fused=max(1, int(kmap[str(c.n)]))))):
            plans = [qsim.Plan(c, qsim.C64, use_graph=True, **mk(c)) for c in cs]
            def run_all(keep=None):
                for i, (c, p) in enumerate(zip(cs, plans)):
                    st = states[c.n]
                    st.set_basis(0)
                    p.execute(st)
                    z = st.expect_z()
                    if keep is not None:
                        keep.append(z)
            run_all()
            torch.cuda.synchronize()
            t = time.perf_counter()
            zs = []
            run_all(zs)
            torch.cuda.synchronize()
            sec = time.perf_counter() - t
            dz = max(float(np.max(np.abs(zs[i][0] - res[i][0]))) for i in range(len(cs)))
            one_by_one[name] = {"ms": sec * 1000.0, "gates_per_s": gates / sec,
                                "passes": sum(p.info["passes"] for p in plans),
                                "max_abs_diff_zi_vs_batch": dz}
            for p in plans:
                p.close()
        for st in states.values():
            st.close()
    line = _common_line(f"gate-applications/s, batch of {len(cs)} TFIM chains (10-{args.nmax} qubits, 8-32 Trotter "
                        "steps), complex64, one persistent launch", gates / (ms / 1000.0), UNIT, args, ms, "f32",
                        {"workload": f"{len(cs)} TFIM chains seed 4, {gates} gates, "
                                     f"{sum(1 for c in cs if c.n > 13)} circuits > 13 qubits",
                         "fusion_k_by_width": kmap, "passes": b.info["passes"],
                         "tensor_core_plans": f"{sum(1 for c in cs if c.n >= tc_min_n)} circuits of >= {tc_min_n} "
                                              f"qubits, {'3xTF32 k = 6' if tc_prec == 1 else 'FP16X3 k <= 7'}, "
                                              f"{b.info['tc_blocks']} blocks",
                         "ms_by_wide_precision": wide_ms},
                        circuits_per_s=len(cs) / (ms / 1000.0),
                        roofline={"bound": "hbm", "achieved": gbs, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                                  "frac": gbs / peaks["hbm_gbs"], "traffic": None, "kernel": "k_batch + k_tc_block",
                                  "note": "algorithmic bytes of the circuits > 13 qubits only; smaller ones stay "
                                          "in shared memory", "peak_source": src},
                        e2e={"value": gates / e2e_s, "unit": UNIT, "h2d_bytes_per_step":
                             sum(16 * 4 ** len(g.targets) for c in cs for g in c.gates),
                             "d2h_bytes_per_step": 8 * sum(2 * c.n - 1 for c in cs)},
                        tune_s=tune_s, sample_zi0=list(res[0][0][:4]), one_by_one=one_by_one, e2e_breakdown=best,
                        e2e_planned_then_executed=min(staged, key=lambda r: r["total_s"]),
                        own_precision=simt_only)
    if not args.no_cpu:
        import oracle as oracle_mod
        # oracle on the smallest circuits until the time budget runs out; work ~ gates x 2^n
        order = sorted(range(len(cs)), key=lambda i: cs[i].n)
        done_work, t0, used = 0.0, time.perf_counter(), 0
        for i in order:
            psi = oracle_mod.run(cs[i])
            oracle_mod.expect_z_chain(psi, cs[i].n)
            done_work += len(cs[i]) * 2.0 ** cs[i].n
            used += 1
            if time.perf_counter() - t0 > args.cpu_seconds:
                break
        dt = time.perf_counter() - t0
        total_work = sum(len(c) * 2.0 ** c.n for c in cs)
        est = dt * total_work / done_work
        line["cpu_baseline"] = {"value": gates / est, "unit": UNIT, "cores": oracle_mod.num_threads(),
                                "kind": "oracle", "sample": f"{used} smallest circuits in {dt:.1f} s, extrapolated "
                                                            f"to the batch by work = gates x 2^n"}
        # accuracy: <Z_i>, <Z_i Z_i+1> of the circuits the oracle ran, plus the two shortest circuits among
        # those planned for the tensor cores (>= tc_min_n qubits), against the oracle's
        wide = sorted((i for i in range(len(cs)) if cs[i].n >= tc_min_n), key=lambda i: len(cs[i]) * 2.0 ** cs[i].n)[:2]
        dzi = dzz = 0.0
        for i in order[:used] + wide:
            zi_r, zz_r = oracle_mod.expect_z_chain(oracle_mod.run(cs[i]), cs[i].n)
            dzi = max(dzi, float(np.max(np.abs(res[i][0] - zi_r))))
            dzz = max(dzz, float(np.max(np.abs(res[i][1] - zz_r)))) if cs[i].n > 1 else dzz
        line["accuracy_vs_oracle"] = {"max_abs_dzi": dzi, "max_abs_dzz": dzz, "circuits": used + len(wide),
                                      "widths": sorted({cs[i].n for i in order[:used] + wide}),
                                      "tensor_core_circuits": [cs[i].n for i in wide]}
    print(json.dumps(line))
    return 0


def run_pairs34(args):
    """34-qubit complex64 state (128 GiB): 16 layers of Haar U(4) on seeded random matchings (seed 5), the top
    4 qubits treated as global index bits (reorder passes before gates on them, identity order restored at
    the end), then 10^5 samples (seed 6): fused 6-qubit blocks in 3xTF32 and in FP16X3 (the faster is
    reported), and the plain per-gate path. Also timed: the same circuit addressing every qubit in place."""
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    n = args.n if args.n != 30 else 34
    c = W.random_pairs(n, 16, seed=5)
    st = qsim.State(n, qsim.C64)
    out = {}
    L = n - 4
    tc6 = dict(mode=1, max_fused=6, precision=1, tc_min_k=5)
    fp6 = dict(mode=1, max_fused=6, precision=4, tc_min_k=5)
    variants = [("tf32x3_k6_reorder_L%d" % L, dict(tc6, local_qubits=L)),
                ("fp16x3_k6_reorder_L%d" % L, dict(fp6, local_qubits=L)), ("tf32x3_k6_in_place", dict(tc6)),
                ("plain_reorder_L%d" % L, dict(mode=0, max_fused=2, local_qubits=L)),
                ("plain_in_place", dict(mode=0, max_fused=2))]
    if args.no_variants:
        variants = variants[:2]
    for name, kw in variants:
        p = qsim.Plan(c, **kw)
        p.pass_list = p.passes()
        st.set_basis(0)
        p.execute(st)
        st.sample(6, 100000)
        torch.cuda.synchronize()
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(len(p.pass_list) + 2)]
        stream = torch.cuda.current_stream()
        st.set_basis(0)
        evs[0].record(stream)
        for i in range(len(p.pass_list)):
            p.execute_range(st, i, 1)
            evs[i + 1].record(stream)
        smp = st.sample(6, 100000)
        evs[-1].record(stream)
        torch.cuda.synchronize()
        per = [evs[i].elapsed_time(evs[i + 1]) for i in range(len(p.pass_list))]
        total = evs[0].elapsed_time(evs[-1])
        reo = sum(m for m, q in zip(per, p.pass_list) if q["kind"] == "reorder")
        gate_ms = sum(m for m, q in zip(per, p.pass_list) if q["kind"] != "reorder")
        gate_bytes = sum(q["algorithmic_bytes"] for q in p.pass_list if q["kind"] != "reorder")
        reo_bytes = sum(q["algorithmic_bytes"] for q in p.pass_list if q["kind"] == "reorder")
        out[name] = {"ms_total": total, "gates_per_s": len(c) / (total / 1000.0), "passes": len(p.pass_list),
                     "reorder_passes": sum(1 for q in p.pass_list if q["kind"] == "reorder"),
                     "reorder_ms": reo, "reorder_gbs": reo_bytes / (reo / 1000.0) / 1e9 if reo > 0 else None,
                     "gate_pass_gbs": gate_bytes / (gate_ms / 1000.0) / 1e9,
                     "sample_ms": evs[len(p.pass_list)].elapsed_time(evs[-1]), "norm": st.norm()}
        p.close()
    main = min(("tf32x3_k6_reorder_L%d" % L, "fp16x3_k6_reorder_L%d" % L), key=lambda k: out[k]["ms_total"])
    line = _common_line(f"gate-applications/s, {n}-qubit random U(4) pairs depth 16, complex64, reorder passes "
                        f"for {4} global qubits, 1e5 samples", out[main]["gates_per_s"], UNIT, args,
                        out[main]["ms_total"], main[:4],
                        {"workload": f"random pairs n={n} depth 16 seed 5, {len(c)} gates, 1e5 samples seed 6",
                         "path": main},
                        paths=out)
    print(json.dumps(line))
    return 0


def run_paper33(args, kind):
    """The paper's own single-GPU benchmarks at its 33-qubit size (Sec. 3, single-GPU generational speedups):
    QPE with an exactly representable phase (32 counting qubits, so all 1000 shots must return the encoded
    integer), its random-circuit script (30n gates: CZ with probability 0.25, else H / RX / RY / RZ) and a
    TFIM Trotter evolution (Eq. 1) on a 33-site periodic triangular lattice standing in for HamLib's.
    A step is |0...0>, every pass of the plan and 1000 shots, as the paper times a run; the paper runs each
    circuit twice and times the second, which the warm-up step covers. Complex64 (64 GiB state)."""
    import numpy as np
    import torch
    import oracle as oracle_mod
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    n = args.n if args.n != 30 else 33
    shots = 1000
    if kind == "qpe":
        a = W.basis_index(n - 1, 7)
        c, expect_a = W.qpe(n - 1, a)
        expect = expect_a | (1 << (n - 1))  # counting register = a, eigenstate qubit in |1>
        small = lambda m: W.qpe(m - 1, W.basis_index(m - 1, 7))[0]
        context = {"paper_time_s": 0.843, "paper_gates": 625, "hardware": "one GB200 (CUDA-Q, cuQuantum)",
                   "note": "the paper's QPE comes from the QED-C suite; this one is built from the same parts"}
    elif kind == "tfim":
        # a 3 x 11 periodic triangular lattice (33 sites, 99 bonds), 10 first-order Trotter steps
        rng = np.random.default_rng(SEED)
        th, ph = (float(x) for x in rng.uniform(0.0, math.pi, size=2))
        n = 33
        c = W.tfim_lattice(11, 3, 10, th, ph)
        expect = None
        small = lambda m: W.tfim_lattice(8, 3, 10, th, ph)
        context = {"paper_time_s_a100": 71.589, "paper_estimate_s_gb200": round(71.589 / 4.51, 2),
                   "paper_gates": 2987, "note": "HamLib 33-qubit TFIM (its lattice file is not available; its "
                   "ZZ terms are decomposed into CNOT-RZ-CNOT, here native RZZ); A100 time and the paper's "
                   "A100 -> GB200 factor 4.51 for QPE"}
    else:
        c = W.rcs(n, seed=SEED)
        expect = None
        small = lambda m: W.rcs(m, seed=SEED)
        context = {"paper_time_s_a100": 5.907, "paper_estimate_s_gb200": round(5.907 / 4.51, 3),
                   "paper_gates": 30 * n, "note": "A100 time and the paper's A100 -> GB200 factor 4.51 for QPE"}
    st = qsim.State(n, qsim.C64)
    peaks, _ = measured_peaks()
    out = {}
    ref_amps = None
    rng = np.random.default_rng(1)
    ys = torch.from_numpy(np.sort(rng.choice(1 << n, size=4096, replace=False))).cuda()
    for name, kw in [("plain", dict(mode=0, max_fused=1)), ("tf32x3_k5", dict(mode=1, max_fused=5, precision=1, tc_min_k=5)),
                     ("tf32x3_k6", dict(mode=1, max_fused=6, precision=1, tc_min_k=5)),
                     ("tf32x3_k6_lookahead", dict(mode=1, max_fused=6, precision=1, tc_min_k=5, plan_effort=1)),
                     ("bf16x6_k6", dict(mode=1, max_fused=6, precision=3, tc_min_k=5)),
                     ("fp16x3_k6", dict(mode=1, max_fused=6, precision=4, tc_min_k=5)),
                     ("fp16x3_k7", dict(mode=1, max_fused=7, precision=4, tc_min_k=5))]:
        if name == "plain" and args.no_variants:
            continue
        p = qsim.Plan(c, **kw)
        samples = []

        def step(i, p=p):
            st.set_basis(0)
            p.execute(st)
            samples.append(st.sample(SEED + i, shots))
        steps = 1 if name == "plain" else max(1, args.steps)
        for _ in range(1 if name == "plain" else max(1, args.warmup)):
            step(0)
        samples.clear()
        ms = _event_time(torch, step, steps)
        amps = st.tensor[ys].cpu().numpy().astype(np.complex128)
        if ref_amps is None:
            ref_amps = amps
        rec = {"ms_per_step": ms, "gates_per_s": len(c) / (ms / 1000.0), "passes": p.info["passes"],
               "host_plan_ms": p.info["host_plan_ms"],
               "algorithmic_gb": p.info["algorithmic_bytes"] / 1e9,
               "achieved_gbs": p.info["algorithmic_bytes"] / (ms / 1000.0) / 1e9,
               "max_abs_diff_sampled_vs_first": float(np.max(np.abs(amps - ref_amps))), "norm": st.norm()}
        if expect is not None:
            rec["shots_equal_to_encoded_phase"] = int(sum(int(np.sum(s == expect)) for s in samples))
            rec["shots"] = shots * len(samples)
        out[name] = rec
        p.close()
    best = min((k for k in out if k != "plain"), key=lambda k: out[k]["ms_per_step"])
    b = out[best]
    title = {"qpe": "QPE", "rcs": "random circuit (30n gates)",
             "tfim": "TFIM on a periodic triangular lattice (10 Trotter steps)"}[kind]
    desc = {"qpe": lambda: f"QPE, {n - 1} counting qubits, phase {expect_a}/2^{n - 1}",
            "rcs": lambda: f"paper random-circuit script n={n} seed={SEED}",
            "tfim": lambda: f"TFIM 3x11 periodic triangular lattice, 99 bonds, theta={th:.4f} phi={ph:.4f}"}[kind]()
    line = _common_line(f"gate-applications/s, {n}-qubit {title}, complex64, 1000 shots", b["gates_per_s"], UNIT, args,
                        b["ms_per_step"], best[:4], {"workload": desc + f", {len(c)} gates", "path": best, "shots": shots},
                        paths=out, peak_hbm_gbs=peaks["hbm_gbs"], paper_context=context)
    del st
    torch.cuda.empty_cache()
    if not args.no_cpu:
        # the oracle on the same generator at 24 qubits for a bounded time, rate scaled by 2^(24 - n)
        n_s = 24
        cs = small(n_s)
        psi = oracle_mod.basis(n_s, 0)
        t = time.perf_counter()
        g = 0
        for gate in cs.gates:
            oracle_mod.apply_gate(psi, n_s, gate.targets, gate.controls, gate.matrix)
            g += 1
            if time.perf_counter() - t > args.cpu_seconds:
                break
        dt = time.perf_counter() - t
        line["cpu_baseline"] = {"value": g / dt * 2.0 ** (n_s - n), "unit": UNIT, "cores": oracle_mod.num_threads(),
                                "kind": "oracle", "sample": f"first {g} gates of the {n_s}-qubit instance in {dt:.1f} s,"
                                                            f" rate scaled by 2^({n_s}-{n})"}
    print(json.dumps(line))
    return 0


def run_spill(args):
    """A state larger than a device window held in host memory (Sec. 2.5): the 30-qubit-generator brickwork at
    n = 33 (64 GiB complex64, page-locked host memory), streamed through three device windows of 2^28
    amplitudes, fused 3xTF32 blocks in every window. Reports gate-applications/s and the host-link bytes per
    second of the streamed run (both directions counted), beside the same circuit run in device memory."""
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    n = args.n if args.n != 30 else 33
    window = 28
    c = W.brickwork(n, 4, seed=SEED)
    kw = dict(mode=1, max_fused=6, precision=1)
    host = torch.empty(1 << n, dtype=torch.complex64, pin_memory=True)
    runs = []
    for i in range(max(1, args.warmup) + max(1, args.steps)):
        host.zero_()
        host[0] = 1.0
        runs.append(qsim.spill_run(host, c, 0, window_qubits=window, **kw))
    timed = runs[max(1, args.warmup):]
    ms = sum(r["elapsed_ms"] for r in timed) / len(timed)
    gbs = sum(r["host_bytes"] for r in timed) / (sum(r["elapsed_ms"] for r in timed) / 1000.0) / 1e9
    # the link itself: 2 GiB page-locked copies host -> device, device -> host, and both at once (two streams)
    nb = 1 << 28
    hsrc = host[:nb]
    hdst = torch.empty(nb, dtype=torch.complex64, pin_memory=True)
    d0 = torch.empty(nb, dtype=torch.complex64, device="cuda")
    d1 = torch.empty(nb, dtype=torch.complex64, device="cuda")
    s_a, s_b = torch.cuda.Stream(), torch.cuda.Stream()

    def link(h2d, d2h, reps=3):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(reps):
            if h2d:
                with torch.cuda.stream(s_a):
                    d0.copy_(hsrc, non_blocking=True)
            if d2h:
                with torch.cuda.stream(s_b):
                    hdst.copy_(d1, non_blocking=True)
        torch.cuda.synchronize()
        return reps * 8 * nb * (int(h2d) + int(d2h)) / (time.perf_counter() - t) / 1e9
    link(True, True, 1)  # first use of the device buffers and streams, untimed
    link_gbs = {"h2d": link(True, False), "d2h": link(False, True), "both": link(True, True)}
    del d0, d1, hdst
    st = qsim.State(n, qsim.C64)
    p = qsim.Plan(c, qsim.C64, **kw)
    dev_ms = _event_time(torch, lambda i: (st.set_basis(0), p.execute(st)), 2)
    r = timed[-1]
    line = _common_line(f"gate-applications/s, {n}-qubit random brickwork depth 4 held in host memory, streamed "
                        f"through 2^{window}-amplitude device windows", len(c) / (ms / 1000.0), UNIT, args, ms, "tf32",
                        {"workload": f"random brickwork n={n} depth 4 seed={SEED}, {len(c)} gates, complex64, "
                                     f"host state {8 * 2 ** n / 2 ** 30:.0f} GiB page-locked", "path": "tf32x3_k6",
                         "window_qubits": window, "global_slots": r["global_slots"]},
                        segments=r["segments"], windows=r["windows"], passes_per_window=r["passes"] / r["windows"],
                        host_link={"bytes_per_run": r["host_bytes"], "gbs": gbs,
                                   "note": "host<->device bytes / wall time of the streamed run, both directions",
                                   "copy_gbs": link_gbs, "fraction_of_both": gbs / link_gbs["both"]},
                        in_device_ms=dev_ms, plan_ms=r["host_plan_ms"])
    print(json.dumps(line))
    return 0


def run_passes(args):
    """Every pass of the brickwork plan timed on its own (CUDA events around five repeats of the pass, after
    one untimed), for the paths named by --path (comma-separated; default tf32x3,fp16x3,fp16x3_pairs): per pass its kind,
    qubits and milliseconds. A profiling aid: it shows which passes of a plan are slow."""
    import torch
    import workloads as W
    from paper_2511_14664_gb300 import qsim
    n, depth = args.n, args.depth
    c = W.brickwork(n, depth, seed=SEED)
    st = qsim.State(n, qsim.C64)
    paths = ["tf32x3", "fp16x3", "fp16x3_pairs"] if args.path == "auto" else args.path.split(",")
    out = {}
    for name in paths:
        p = make_plan(qsim, c, name)
        ps = p.passes()
        st.set_basis(0)
        p.execute(st)
        torch.cuda.synchronize()
        rows = []
        for i, q in enumerate(ps):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            p.execute_range(st, i, 1)
            e0.record()
            for _ in range(5):
                p.execute_range(st, i, 1)
            e1.record()
            torch.cuda.synchronize()
            rows.append({"kind": q["kind"], "targets": q["targets"], "second": q["controls"] if q["kind"] == "tc_pair" else [],
                         "ms": e0.elapsed_time(e1) / 5})
        out[name] = {"passes": rows, "total_ms": sum(r["ms"] for r in rows)}
        p.close()
    print(json.dumps({"workload": f"random brickwork n={n} depth={depth} seed={SEED}", "per_pass": out}))
    return 0


def main():
    args = parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "qft28":
        return run_qft(args)
    if args.workload == "brick14":
        return run_brick14(args)
    if args.workload == "tfim_batch":
        return run_tfim_batch(args)
    if args.workload == "pairs34":
        return run_pairs34(args)
    if args.workload in ("qpe33", "rcs33"):
        return run_paper33(args, args.workload[:3])
    if args.workload == "tfim33":
        return run_paper33(args, "tfim")
    if args.workload == "spill33":
        return run_spill(args)
    if args.workload == "passes":
        return run_passes(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
