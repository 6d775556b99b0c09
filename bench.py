#!/usr/bin/env python
"""Benchmark of the split-FP16 SP2 solve (Alg. 1 + Eq. 15) on one GB300.

Workload: the large mixed-precision case, N = 16384, N_occ = 8192, spectrum
U[-2, -0.025] U U[0.025, 2], H = Q diag(eps) Q^T with Q from the QR of a
seeded Gaussian matrix (seed 0), stored FP32.  One step = one complete solve
H -> D (Gershgorin bounds, input layer, all squaring layers, refinement).

Printed (one JSON line on rank 0):
  value      effective TFLOP/s = (squaring layers incl. refinement) x 2 N^3 / time-to-D
             (2 N^3 = the work of one dense N x N square; same count for every arm)
  ms_per_step  time-to-D (device time, CUDA events)
  e2e        the same metric through the C ABI with H copied from pinned host
             memory and D copied back inside the timed region
  roofline   the squaring kernel: 3 N^3 algorithmic tensor FLOPs per launch
             (hi hi + hi lo + lo hi over the upper half) / its mean launch time
  cpu_baseline  the FP64 oracle on a bounded sample of the same workload
Also: the plain FP32 (FFMA) path's time-to-D on the same input, and sampled
parity of D against the closed form Q_occ Q_occ^T.

--impl reference times the FP64 CPU oracle itself (one row block of one
layer per step) on the same workload and prints the same line with
"impl": "reference".
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
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

WORKLOAD = dict(N=16384, n_occ=8192, occ=(-2.0, -0.025), virt=(0.025, 2.0), seed=0)
METRIC = "SP2 time-to-D and TFLOP/s at N=16384 vs FP32 path, max-abs err vs FP64 oracle"
FALLBACK_PEAKS = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}


def _args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=WORKLOAD["N"])
    ap.add_argument("--max-iter", type=int, default=100)
    ap.add_argument("--no-fp32", action="store_true", help="skip the FP32 comparator")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU baseline")
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--gen-device", default="gpu", choices=["gpu", "cpu"],
                    help="where the input generator runs its FP64 QR (cpu: for runs under a profiler)")
    ap.add_argument("--input-cache", default=None,
                    help="directory: reuse the generated Hamiltonian (H, Q, eps) stored there by an earlier run, "
                         "else generate and store it (profiled runs then need no QR)")
    ap.add_argument("--cpu-seconds", type=float, default=12.0, help="target length of the CPU sample")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched-SP2 measurement")
    ap.add_argument("--no-network", action="store_true", help="skip the network forward/backward measurement")
    ap.add_argument("--no-accel", action="store_true", help="skip the accelerated-layer measurement")
    ap.add_argument("--only", default=None, choices=["batched", "network", "fermi"],
                    help="run one secondary measurement alone and print it (profiling runs)")
    ap.add_argument("--batched-count", type=int, default=512)
    return ap.parse_args()


def _workload(n):
    w = dict(WORKLOAD)
    if n != w["N"]:
        w["N"], w["n_occ"] = n, n // 2
    return w


def _cached_input(cache_dir, w, make):
    """The workload's Hamiltonian, from cache_dir when an earlier run stored
    it there (same N, occupation, spectrum intervals and seed), else made
    and, with a cache_dir, stored."""
    if not cache_dir:
        return make()
    import sp2_inputs

    key = f"sp2_input_N{w['N']}_occ{w['n_occ']}_{w['occ'][0]}_{w['occ'][1]}_{w['virt'][0]}_{w['virt'][1]}_s{w['seed']}"
    path = os.path.join(cache_dir, key + ".npz")
    if os.path.exists(path):
        z = np.load(path)
        return sp2_inputs.Hamiltonian(H=z["H"], Q=z["Q"], eps=z["eps"], n_occ=int(z["n_occ"]), seed=int(z["seed"]))
    h = make()
    os.makedirs(cache_dir, exist_ok=True)
    np.savez(path, H=h.H, Q=h.Q, eps=h.eps, n_occ=h.n_occ, seed=h.seed)
    return h


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d, "measured"
    return FALLBACK_PEAKS, "fallback"


def replica_time_max(ms, dev, ws):
    """Whole-job time of N independent replicas: the slowest rank's time
    (all-reduce MAX over the process group; identity on one rank)."""
    if ws <= 1:
        return ms
    import torch
    import torch.distributed as dist

    t = torch.tensor([float(ms)], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(units_per_rank, ms, ws):
    """Aggregate rate of ws replicas that each processed units_per_rank in the
    whole-job time ms (weak scaling: per-rank work fixed)."""
    return units_per_rank * ws / (ms * 1e-3)


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class Clocks:
    """nvidia-smi sampler running during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(prefix="sp2clk", suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons, pw = [], None, set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as f:
            for line in f:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    smax = float(parts[2])
                except ValueError:
                    continue
                try:
                    pw.append(float(parts[3]))
                except ValueError:
                    pass
                for nm, v in zip(names, parts[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(nm)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm),
                "power_w": statistics.median(pw) if pw else None}


# sources that define the timed squaring kernel; the committed DRAM-traffic
# figure is used only while their combined hash matches the one it was taken on
KERNEL_SOURCES = ["syrk_tc2.cu", "epilogue.cuh", "tc_ptx.cuh", "tile_finish.cuh", "common.cuh", "kernels.h"]


def kernel_source_hash():
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        h.update(open(os.path.join(ROOT, "paper_2101_06385_gb300", "csrc", f), "rb").read())
    return h.hexdigest()


def _traffic_from_profile(n):
    """DRAM bytes per launch of the squaring kernel from the committed ncu
    summary, if it was taken on the current kernel source."""
    prof = os.path.join(ROOT, "profiles", "syrk_tc2_split_n16384.md")
    if not os.path.exists(prof) or n != WORKLOAD["N"]:
        return None
    text = open(prof).read()
    m = re.search(r"kernel_source_sha256:\s*([0-9a-f]{64})", text)
    t = re.search(r"dram_bytes_per_launch_n16384:\s*([0-9.eE+]+)", text)
    if not m or not t:
        return None
    return float(t.group(1)) if kernel_source_hash() == m.group(1) else None


def energy_of(power_w, ms_per_solve, layers):
    """Energy of one solve and one squaring layer from the median board power
    sampled during the timed region (None when no power was sampled)."""
    if not power_w or not ms_per_solve or not layers:
        return None
    j = power_w * ms_per_solve * 1e-3
    return {"power_w_median": power_w, "joules_per_solve": j, "joules_per_layer": j / layers}


def _oracle_one_core(n=4096, rows=256):
    """The oracle's layer sample on one core: a child process whose BLAS and
    OpenMP pools are pinned to one thread before numpy loads; a seeded dense
    symmetric n x n matrix, ``rows`` rows of the product."""
    code = (
        "import json, time, numpy as np, oracle\n"
        f"rng = np.random.default_rng(0); A = rng.uniform(-1, 1, ({n}, {n})); S = (A + A.T) / 2\n"
        f"oracle.sp2_layer_sample(S, 64)\n"
        f"t = time.perf_counter(); oracle.sp2_layer_sample(S, {rows}); dt = time.perf_counter() - t\n"
        f"print(json.dumps({{'value': 2.0 * {rows} * {n} ** 2 / dt / 1e12, 'unit': 'TFLOP/s', "
        f"'sample': 'one FP64 layer, {rows} of {n} rows', 'seconds': dt}}))\n")
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "BLIS_NUM_THREADS"):
        env[k] = "1"
    env["PYTHONPATH"] = ROOT + os.pathsep + env.get("PYTHONPATH", "")
    try:
        r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
        return json.loads(r.stdout.strip().splitlines()[-1]) if r.returncode == 0 else None
    except (subprocess.SubprocessError, ValueError, IndexError):
        return None


def _cpu_model():
    try:
        for line in open("/proc/cpuinfo"):
            k = line.split(":")[0].strip().lower()
            if k in ("model name", "cpu model", "hardware"):
                return line.split(":", 1)[1].strip()
        import platform

        return platform.processor() or platform.machine()
    except OSError:
        return None


def _cpu_threads():
    try:
        from threadpoolctl import threadpool_info

        n = [i.get("num_threads") for i in threadpool_info() if i.get("user_api") == "blas"]
        if n:
            return int(max(n))
    except Exception:
        pass
    return os.cpu_count()


def _oracle_sample(H64, w, target_s):
    """FP64 oracle on a bounded sample: Gershgorin + input layer, then one
    layer restricted to a block of rows, sized to take about target_s."""
    import oracle

    N = w["N"]
    t0 = time.perf_counter()
    lo, hi = oracle.gershgorin_bounds(H64)
    S0 = oracle.input_layer(H64, lo, hi)
    t_pro = time.perf_counter() - t0
    rows = 256
    t0 = time.perf_counter()
    oracle.sp2_layer_sample(S0, rows)
    dt = time.perf_counter() - t0
    rows = int(min(N, max(256, rows * target_s / max(dt, 1e-3))))
    rows = max(256, rows // 256 * 256)
    return S0, rows, t_pro


def run_reference(args):
    import torch

    ws, rank, local = _dist()
    if rank != 0:
        return 0
    w = _workload(args.n)
    import sp2_inputs

    dev = "cuda" if torch.cuda.is_available() else "cpu"
    h = sp2_inputs.gapped_hamiltonian(w["N"], w["n_occ"], w["occ"], w["virt"], w["seed"], device=dev)
    H64 = h.H.astype(np.float32).astype(np.float64)
    del h
    import oracle

    S0, rows, _ = _oracle_sample(H64, w, max(2.0, min(args.cpu_seconds, 20.0)))
    N = w["N"]
    for _ in range(args.warmup):
        oracle.sp2_layer_sample(S0, rows)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.sp2_layer_sample(S0, rows)
    dt = (time.perf_counter() - t0) / args.steps
    flops = 2.0 * rows * N * N
    value = flops / dt / 1e12
    cores = _cpu_threads()
    sample = f"one SP2 layer (S[:{rows}] @ S, update, trace) of the N={N} workload per step, FP64 numpy"
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "TFLOP/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"sp2_dense_gapped_N{N}_nocc{w['n_occ']}", "N": N, "n_occ": w["n_occ"],
                   "flop_convention": "2N^3 per squaring layer (dense-square equivalent)",
                   "l2": "inputs (1 GiB FP32 H) larger than L2"},
        "cpu_baseline": {"value": value, "unit": "TFLOP/s", "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": "TFLOP/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


def _bench_batched(sp2, sp2_inputs, dev, reps=3, count=512):
    """512 Hamiltonians, N uniform in {64..1024} step 32, gaps U[0.05, 0.3]."""
    import torch

    cfg = sp2_inputs.batched_config(count=count)
    Hs = [torch.from_numpy(sp2_inputs.batched_instance(N, n, g, s).h32()).to(dev) for (N, n, g, s) in cfg]
    n_occ = [c[1] for c in cfg]
    sp2.density_matrix_batched(Hs, n_occ)
    torch.cuda.synchronize(dev)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        _, st = sp2.density_matrix_batched(Hs, n_occ)
    e1.record()
    torch.cuda.synchronize(dev)
    ms = e0.elapsed_time(e1) / reps
    layers = [s.iterations + 2 for s in st]
    flops = sum(l * 2.0 * c[0] ** 3 for l, c in zip(layers, cfg))
    alg = sum(l * 3.0 * c[0] ** 3 for l, c in zip(layers, cfg))
    # per-instance accuracy on a seeded sample of instances: the whole D
    # against Q_occ Q_occ^T of the generator (Eq. 6), outside the timed region
    Ds, _ = sp2.density_matrix_batched(Hs, n_occ)
    torch.cuda.synchronize(dev)
    pick = np.random.default_rng(5).choice(len(cfg), size=min(16, len(cfg)), replace=False)
    errs, tr_errs = [], []
    for i in sorted(pick):
        N, n, g, sd = cfg[i]
        h = sp2_inputs.batched_instance(N, n, g, sd)
        Qo = h.Q[:, :n]
        Di = Ds[i].cpu().numpy().astype(np.float64)
        errs.append(float(np.max(np.abs(Di - Qo @ Qo.T))))
        tr_errs.append(abs(float(np.trace(Di)) - n))
    return {"instances": len(cfg), "ms": ms, "tflops_2n3": flops / (ms * 1e-3) / 1e12,
            "tflops_split_alg_3n3": alg / (ms * 1e-3) / 1e12, "layers_min": min(layers),
            "layers_mean": float(np.mean(layers)), "layers_max": max(layers),
            "all_converged": all(s.status == 0 for s in st),
            "accuracy": {"instances_checked": len(errs), "sizes": [int(cfg[i][0]) for i in sorted(pick)],
                         "max_abs_err_worst": max(errs), "max_abs_err_median": float(np.median(errs)),
                         "trace_err_worst": max(tr_errs), "reference": "closed form Q_occ Q_occ^T, whole D"}}


def _bench_network(sp2, sp2_inputs, dev, B=64, N=2048, L=20, ckpt_every=5, reps=2, grad_check=True, gen="gpu"):
    """Differentiable network: 64 gapped Hamiltonians of N = 2048, 20 layers,
    coefficients initialised to the SP2 branch values of instance 0."""
    import torch

    hs = [sp2_inputs.gapped_hamiltonian(N, N // 2, (-1.0, -0.05), (0.05, 1.0), 2000 + i,
                                        device=str(dev) if gen == "gpu" else "cpu")
          for i in range(B)]
    H = torch.from_numpy(np.stack([x.h32() for x in hs])).to(dev)
    _, st = sp2.density_matrix(H[0].contiguous(), N // 2, precision="split")
    sig = st.sigmas + [1 if k % 2 == 0 else -1 for k in range(L)]
    coef = torch.tensor([[1.0, 0.0, 0.0] if s > 0 else [-1.0, 2.0, 0.0] for s in sig[:L]], dtype=torch.float32)
    X, ck, _ = sp2.network_forward(H, coef, ckpt_every)
    G = torch.randn_like(X) * 1e-3
    G = 0.5 * (G + G.transpose(1, 2))
    sp2.network_backward(H, coef, ckpt_every, ck, G.contiguous())
    torch.cuda.synchronize(dev)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    ev[0].record()
    for _ in range(reps):
        X, ck, _ = sp2.network_forward(H, coef, ckpt_every)
    ev[1].record()
    for _ in range(reps):
        sp2.network_backward(H, coef, ckpt_every, ck, G.contiguous())
    ev[2].record()
    torch.cuda.synchronize(dev)
    fwd = ev[0].elapsed_time(ev[1]) / reps
    bwd = ev[1].elapsed_time(ev[2]) / reps
    f_fwd = B * L * 3.0 * N ** 3
    # backward: recomputation of the non-checkpointed layers + the split SYR2K (6 N^3 per layer)
    f_bwd = B * (L - (L + ckpt_every - 1) // ckpt_every) * 3.0 * N ** 3 + B * L * 6.0 * N ** 3
    out = {"B": B, "N": N, "layers": L, "ckpt_every": ckpt_every, "forward_ms": fwd, "backward_ms": bwd,
           "forward_tflops_alg": f_fwd / (fwd * 1e-3) / 1e12, "backward_tflops_alg": f_bwd / (bwd * 1e-3) / 1e12}
    if grad_check:
        out["gradient_check"] = _network_grad_check(sp2, sp2_inputs, dev, H, hs, coef, ckpt_every)
    return out


def _network_grad_check(sp2, sp2_inputs, dev, H, hs, coef, ckpt_every, sub=2, h=1e-4):
    """Gradient errors of the network (outside any timed region), with the
    loss of reading C16 against the Fermi-Dirac target (kT = 0.05, mu = 0):
    (a) the adjoint's dL/dcoef on the whole batch against central differences
    of the GPU forward (loss summed in FP64) on six coefficients; (b) the
    adjoint on a sub-batch against the FP64 oracle's adjoint (the oracle is
    test infrastructure: a CPU reference, not part of the timed path)."""
    import torch

    import oracle

    B, N = H.shape[0], H.shape[1]
    L = coef.shape[0]
    T = torch.empty((B, N, N), dtype=torch.float64, device=dev)
    for b, x in enumerate(hs):
        Q = torch.from_numpy(x.Q).to(dev)
        occ = 1.0 / (1.0 + torch.exp(torch.from_numpy(x.eps).to(dev) / 0.05))
        T[b] = (Q * occ[None, :]) @ Q.T
    del Q
    X, ck, _ = sp2.network_forward(H, coef, ckpt_every)
    G_L = (2.0 * (X.double() - T) / B).float().contiguous()
    dcoef, _ = sp2.network_backward(H, coef, ckpt_every, ck, G_L)
    d = dcoef.numpy().astype(np.float64)

    def loss(cf):
        Xc, _, _ = sp2.network_forward(H, cf, ckpt_every)
        return float(((Xc.double() - T) ** 2).sum().item() / B)

    c32 = coef.numpy().astype(np.float32)
    fd_errs = []
    for n, k in [(0, 0), (0, 1), (L // 4, 2), (L // 2, 0), (3 * L // 4, 1), (L - 1, 2)]:
        cp, cm = c32.copy(), c32.copy()
        cp[n, k] = np.float32(c32[n, k] + h)
        cm[n, k] = np.float32(c32[n, k] - h)
        fd = (loss(torch.from_numpy(cp)) - loss(torch.from_numpy(cm))) / (float(cp[n, k]) - float(cm[n, k]))
        fd_errs.append(abs(fd - d[n, k]) / np.max(np.abs(d)))
    del X, ck, G_L
    # (b) sub-batch against the FP64 oracle adjoint
    Hs = H[:sub].contiguous()
    Xs, cks, _ = sp2.network_forward(Hs, coef, ckpt_every)
    X0 = []
    for x in hs[:sub]:
        H64 = x.h32().astype(np.float64)
        lo, hi = oracle.gershgorin_bounds(H64)
        X0.append(oracle.input_layer(H64, lo, hi))
    X0 = np.stack(X0)
    Ts = T[:sub].cpu().numpy()
    GLs = (2.0 * (Xs.cpu().numpy().astype(np.float64) - Ts) / sub).astype(np.float32)
    ds, G0 = sp2.network_backward(Hs, coef, ckpt_every, cks, torch.from_numpy(GLs).to(dev))
    want_d, want_G0 = oracle.network_adjoint(X0, coef.numpy().astype(np.float64), GLs.astype(np.float64))
    return {"fd_step": h, "fd_coefficients": 6,
            "dcoef_err_vs_central_differences_rel_to_max": float(max(fd_errs)),
            "oracle_sub_batch": sub,
            "dcoef_err_vs_fp64_adjoint_rel_to_max": float(np.max(np.abs(ds.numpy() - want_d)) / np.max(np.abs(want_d))),
            "dX0_err_vs_fp64_adjoint_rel_to_max": float(np.max(np.abs(G0.cpu().numpy() - want_G0))
                                                     / np.max(np.abs(want_G0))),
            "loss": "(1/B) sum ||X_L - D_FD||_F^2, D_FD at kT = 0.05, mu = 0"}


def _bench_fermi(sp2, sp2_inputs, dev, B=64, N=2048, L=11, reps=3, gen="gpu"):
    """Finite-temperature expansion (11 generalised layers with the readout
    fused into the squaring epilogue) on the network workload's 64 instances
    of N = 2048.  The timing does not depend on the coefficient values; the
    SP2 branch polynomials with the readout on the last layer are used."""
    import torch

    Hs = [sp2_inputs.gapped_hamiltonian(N, N // 2, (-1.0, -0.05), (0.05, 1.0), 2000 + i,
                                        device=str(dev) if gen == "gpu" else "cpu").h32()
          for i in range(B)]
    H = torch.from_numpy(np.stack(Hs)).to(dev)
    theta = np.array([[1.0, 0.0, 0.0] if n % 2 else [-1.0, 2.0, 0.0] for n in range(L)])
    c = np.zeros(L + 1)
    c[-1] = 1.0
    D, _ = sp2.fermi_expansion(H, theta, c)
    torch.cuda.synchronize(dev)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        sp2.fermi_expansion(H, theta, c, out=D)
    e1.record()
    torch.cuda.synchronize(dev)
    ms = e0.elapsed_time(e1) / reps
    return {"B": B, "N": N, "layers": L, "ms": ms, "tflops_alg": B * L * 3.0 * N ** 3 / (ms * 1e-3) / 1e12}


def run_ours(args):
    import torch

    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist

        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device("cuda", local if ws > 1 else 0)
    torch.cuda.set_device(dev)
    import paper_2101_06385_gb300 as sp2
    import sp2_inputs

    w = _workload(args.n)
    N, n_occ = w["N"], w["n_occ"]
    t_gen = time.perf_counter()
    gen_dev = str(dev) if args.gen_device == "gpu" else "cpu"
    h = _cached_input(args.input_cache, w, lambda: sp2_inputs.gapped_hamiltonian(
        N, n_occ, w["occ"], w["virt"], w["seed"], device=gen_dev))
    t_gen = time.perf_counter() - t_gen
    H32 = h.h32()
    H = torch.from_numpy(H32).to(dev)
    D = torch.empty_like(H)
    sp2.init(dev.index, precision="split")

    def barrier():
        torch.cuda.synchronize(dev)
        if ws > 1:
            torch.distributed.barrier()

    for _ in range(args.warmup):
        sp2.density_matrix(H, n_occ, max_iter=args.max_iter, out=D, precision="split")
    clk = Clocks(dev.index if dev.index is not None else 0)
    barrier()
    clk.start()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    stats = []
    e0.record()
    for _ in range(args.steps):
        _, st = sp2.density_matrix(H, n_occ, max_iter=args.max_iter, out=D, precision="split")
        stats.append(st)
    e1.record()
    barrier()
    clocks = clk.stop()
    ms = replica_time_max(e0.elapsed_time(e1) / args.steps, dev, ws)
    st = stats[-1]
    layers = st.iterations + 2
    flops_eff = layers * 2.0 * N ** 3
    value = replica_throughput(flops_eff, ms, ws) / 1e12

    # squaring layers of the timed steps; layer slots past a solve's last one take
    # time only where every slot is a launch of its own
    act = [x for s in stats for x in s.square_ms[: s.iterations + 2]]
    idle = [x for s in stats for x in s.square_ms[s.iterations + 2:] if x > 0]
    launch_ms = statistics.mean(act)
    alg_flops = 3.0 * N ** 3
    peaks, src = _peaks()
    peak = float(peaks.get("bf16_tflops_sustained", peaks.get("bf16_tflops")))
    achieved = alg_flops / (launch_ms * 1e-3) / 1e12
    T = (N + 255) // 256
    exec_flops = 2.0 * 128 * 256 * 3 * N * (T * (T + 1))  # two 128x256 CTA tiles per upper 256x256 super tile
    traffic = _traffic_from_profile(N)

    # sampled check of D against the generator's eigenvectors (D_ij = sum over
    # occupied k of Q_ik Q_jk); the full-size parity test lives in tests/
    rng = np.random.default_rng(123)
    ii = rng.integers(0, N, 4096)
    jj = rng.integers(0, N, 4096)
    dd = rng.integers(0, N, 256)
    Dh = D.cpu().numpy()
    want = np.einsum("ik,ik->i", h.Q[ii, :n_occ], h.Q[jj, :n_occ])
    want_d = np.einsum("ik,ik->i", h.Q[dd, :n_occ], h.Q[dd, :n_occ])
    diff = np.concatenate([Dh[ii, jj] - want, Dh[dd, dd] - want_d])
    ref = np.concatenate([want, want_d])
    max_abs = float(np.max(np.abs(diff)))
    rel_frob = float(np.sqrt(np.mean(diff ** 2) / max(np.mean(ref ** 2), 1e-300)))
    trace_err = abs(float(np.trace(Dh.astype(np.float64))) - n_occ)
    # idempotency and commutator with H on 256 sampled rows (FP32 products on
    # the device, outside the timed region)
    with torch.no_grad():
        rr = torch.from_numpy(np.sort(rng.choice(N, 256, replace=False))).to(dev)
        prev_tf32 = torch.backends.cuda.matmul.allow_tf32
        torch.backends.cuda.matmul.allow_tf32 = False
        Dr, Hr = D.index_select(0, rr), H.index_select(0, rr)
        idem = float((Dr @ D - Dr).abs().max())
        comm = float((Dr @ H - Hr @ D).abs().max())
        torch.backends.cuda.matmul.allow_tf32 = prev_tf32

    # FP32 (FFMA) comparator on the same input
    fp32 = None
    if not args.no_fp32:
        Df = torch.empty_like(H)
        sp2.density_matrix(H, n_occ, max_iter=args.max_iter, out=Df, precision="fp32")
        torch.cuda.synchronize(dev)
        _, sf = sp2.density_matrix(H, n_occ, max_iter=args.max_iter, out=Df, precision="fp32")
        Dfh = Df.cpu().numpy()
        fdiff = np.concatenate([Dfh[ii, jj] - want, Dfh[dd, dd] - want_d])
        fp32 = {"time_to_D_ms": sf.time_ms, "layers": sf.iterations + 2,
                "speedup_split_vs_fp32": sf.time_ms / ms,
                "max_abs_err_sampled": float(np.max(np.abs(fdiff)))}
        del Df
        sp2.set_precision("split")

    # end to end through the C ABI: pinned host H -> device -> solve -> host D
    Hh = torch.from_numpy(H32).pin_memory()
    Dhost = torch.empty_like(Hh).pin_memory()
    Hd = torch.empty_like(H)
    s0 = torch.cuda.Event(enable_timing=True)
    s1 = torch.cuda.Event(enable_timing=True)
    barrier()
    s0.record()
    e2e_layers = 0
    for _ in range(args.e2e_steps):
        Hd.copy_(Hh, non_blocking=True)
        _, se = sp2.density_matrix(Hd, n_occ, max_iter=args.max_iter, out=D, precision="split")
        Dhost.copy_(D, non_blocking=True)
        e2e_layers += se.iterations + 2
    s1.record()
    barrier()
    e2e_ms = replica_time_max(s0.elapsed_time(s1) / args.e2e_steps, dev, ws)
    e2e_value = replica_throughput((e2e_layers / args.e2e_steps) * 2.0 * N ** 3, e2e_ms, ws) / 1e12

    cpu = None
    if not args.no_cpu and rank == 0 and ws == 1:
        import oracle

        H64 = H32.astype(np.float64)
        S0, rows, t_pro = _oracle_sample(H64, w, args.cpu_seconds)
        t0 = time.perf_counter()
        oracle.sp2_layer_sample(S0, rows)
        dt = time.perf_counter() - t0
        one_core = _oracle_one_core()
        cpu = {"value": 2.0 * rows * N * N / dt / 1e12, "unit": "TFLOP/s", "cores": _cpu_threads(),
               "kind": "oracle", "cpu_model": _cpu_model(), "one_core": one_core,
               "sample": f"one FP64 SP2 layer restricted to {rows} of {N} rows (S[:rows] @ S + update + trace), "
                         f"{dt:.1f} s; full solve would be ~{layers} layers x {N // rows} blocks"}
        del S0, H64

    # accelerated layers (HOMO/LUMO known, e.g. from a previous MD step): the
    # generator's exact band edges
    accel = None
    if not args.no_accel:
        homo, lumo = float(h.eps[:n_occ].max()), float(h.eps[n_occ:].min())
        sp2.density_matrix_accelerated(H, n_occ, homo, lumo, out=D)
        torch.cuda.synchronize(dev)
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a0.record()
        for _ in range(3):
            _, sa = sp2.density_matrix_accelerated(H, n_occ, homo, lumo, out=D)
        a1.record()
        torch.cuda.synchronize(dev)
        ams = a0.elapsed_time(a1) / 3
        Da = D.cpu().numpy()
        adiff = np.concatenate([Da[ii, jj] - want, Da[dd, dd] - want_d])
        accel = {"time_to_D_ms": ams, "layers": sa.iterations, "speedup_vs_trace_rule": ms / ams,
                 "max_abs_err_sampled": float(np.max(np.abs(adiff))),
                 "trace_err": abs(float(np.trace(Da.astype(np.float64))) - n_occ),
                 "homo_lumo": "exact band edges of the generated spectrum"}
        del Da

    batched = None if args.no_batched else _bench_batched(sp2, sp2_inputs, dev)
    network = None if args.no_network else _bench_network(sp2, sp2_inputs, dev)
    fermi = None if args.no_network else _bench_fermi(sp2, sp2_inputs, dev)

    # Gershgorin, input layer and its row norms, then all layers in one launch (or
    # one launch per layer slot, whose idle ones then show a time)
    launches_per_step = 3 + (st.launches if idle else 1)
    line = {
        "metric": METRIC, "value": value, "unit": "TFLOP/s", "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f16",
        "data": "synthetic (seeded gapped Hamiltonian, dense QR eigenvectors)",
        "config": {"workload": f"sp2_dense_gapped_N{N}_nocc{n_occ}", "N": N, "n_occ": n_occ,
                   "spectrum": "U[-2,-0.025] U U[0.025,2]", "seed": w["seed"],
                   "precision": "split-FP16 (hi + 2^-11 lo) tcgen05 products, FP32 accumulation/storage, "
                                "FP64 bounds/traces/control, alpha*I shift",
                   "flop_convention": "value: 2N^3 per squaring layer incl. 2 refinement layers (dense-square "
                                      "equivalent); roofline: 3N^3 per split layer (upper half)",
                   "parallelism": "replicas" if ws > 1 else "single GPU",
                   "l2": "no flush: inputs (1 GiB FP32 H, 1.5 GiB iterate + splits) larger than L2",
                   "time_to_D_ms": ms, "layers": layers, "loop_layers": st.iterations,
                   "prologue_ms": st.prologue_ms,
                   "converged_by": st.converged_by, "generator_s": round(t_gen, 1),
                   "paper_convention_tflops": st.iterations * 4.0 * N ** 3 / (sum(
                       st.layer_ms[: st.iterations]) * 1e-3) / 1e12},
        "accuracy": {"max_abs_err_sampled": max_abs, "rel_frob_sampled": rel_frob, "trace_err": trace_err,
                     "idempotency_max_abs_sampled_rows": idem, "commutator_max_abs_sampled_rows": comm,
                     "idemp_err_last_layer": st.idemp_err,
                     "samples": int(len(diff)), "tolerance_max_abs": 5e-5, "tolerance_trace": 1e-4},
        "fp32_path": fp32,
        "e2e": {"value": e2e_value, "unit": "TFLOP/s", "ms_per_step": e2e_ms,
                "h2d_bytes_per_step": int(N * N * 4), "d2h_bytes_per_step": int(N * N * 4)},
        "roofline": {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                     "frac": achieved / peak, "traffic": traffic,
                     "peak_source": f"{src} bf16_tflops_sustained (FP16 dense = BF16 dense rate)",
                     "kernel": "syrk_tc2_kernel<split> (CTA pairs, all layers in one launch; wide units at N = 16384)", "launch_ms_mean": launch_ms,
                     "idle_launch_ms_mean": statistics.mean(idle) if idle else None,
                     "executed_tflops": exec_flops / (launch_ms * 1e-3) / 1e12},
        "accelerated": accel,
        "batched": batched,
        "network": network,
        "fermi_expansion": fermi,
        "cpu_baseline": cpu,
        "clocks": clocks,
        # board power sampled during the timed solves and the energy it implies
        "energy": energy_of(clocks.get("power_w"), ms, layers),
        "gpu_launches": int(launches_per_step * args.steps),
    }
    if rank == 0:
        print(json.dumps(line))
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def run_only(args):
    import torch

    import paper_2101_06385_gb300 as sp2
    import sp2_inputs

    dev = torch.device("cuda", 0)
    sp2.init(0, precision="split")
    if args.only == "batched":
        out = _bench_batched(sp2, sp2_inputs, dev, reps=max(1, args.steps), count=args.batched_count)
    elif args.only == "fermi":
        out = _bench_fermi(sp2, sp2_inputs, dev, reps=max(1, args.steps), gen=args.gen_device)
    else:
        out = _bench_network(sp2, sp2_inputs, dev, reps=max(1, args.steps), gen=args.gen_device)
    print(json.dumps({"only": args.only, **out}))
    return 0


def main():
    args = _args()
    if args.impl == "reference":
        return run_reference(args)
    if args.only:
        return run_only(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
