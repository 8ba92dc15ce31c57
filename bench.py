#!/usr/bin/env python
"""Benchmark of the PRISM fit on one GB300 (or N, one process per GPU).

Workload: the HCP-shaped whole brain -- 145 x 174 x 145 grid, ellipsoid mask of
740,110 voxels, 288 measurements (18 b=0 + 90 at each of b = 1000/2000/3000),
SNR 30 Rician, K = 3, MSE, repulsion + sparsity + neighbour coherence (Huber-
Laplacian and directional continuity) inside mask-cropped 16^3 patches. One step
= one iteration of the fit over the whole volume: synthesis, calibration-free
MSE, hand-written adjoint, priors and the Adam update of every parameter, in the
fused persistent kernel replayed from a CUDA graph.

Under torchrun with N ranks (one per GPU) the brain's 16^3 patches are split across the
ranks, balanced by voxel count, each rank fitting its share with the whole brain's |M| as
the normaliser and no collective on the data path (strong scaling: the work is one brain
whatever N is). Prints one JSON line (rank 0). `--impl reference` times the FP64 CPU oracle
on a bounded sample of the same workload instead.
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
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "voxel-iterations/s fused fwd+adjoint+Adam vs unfused, same GB300; % of roofline"
UNIT = "voxel-iterations/s"
WORKLOAD = "hcp_shaped_brain_145x174x145_ellipsoid_mask_N288_K3_mse_patch16"
K_FIB = 3
PRIORS = dict(lam_rep=0.01, lam_sparse=0.02, lam_sp=0.01, lam_dir=0.005)

# FP32 floating-point operations per (voxel, measurement) pair of the fused kernel's loop on
# this workload (MSE, no calibration), fused multiply-add = 2.
# Shell loop (every shell of the scheme even): per fiber 26 -- scaled cosine c' = d . g' 5,
# exponent arguments 2 + 2, f_in e1 + (1 - f_in) p 1, its product with -S0 f_k into the residual
# 2, the two adjoint sums 4, dE/dc factor f_in e1 + rho (1 - f_in) p 2, its product with r c' 2,
# the direction sum 6 -- and per measurement 4 (y - S0 T0 1, the residual's square 2, the
# shell's sum of r 1); the isotropic terms are formed once per shell.
FLOPS_PER_PAIR_SHELL = 4 + 26 * K_FIB
# Per-measurement loop: 17 per measurement (isotropic mixture 5, residual 2, its square 2,
# isotropic adjoint 6, two derivative constants 2) + 28 per fiber.
FLOPS_PER_PAIR = 17 + 28 * K_FIB
# Measurements with b = 0 (leading the table) need no fiber terms: r = y - S0 sum(f) and r^2
# (two multiply-adds) and the running sum of r (one add); in the shell loop r = y + (-S0 T0) is
# one add.
FLOPS_PER_B0_PAIR = 5
FLOPS_PER_B0_PAIR_SHELL = 4
# DRAM bytes per voxel-iteration of the fused kernel (read + write) from an ncu capture of the
# scaled brain (traffic grows in proportion to the voxels), valid only for the kernel sources
# whose SHA-256 (comments and blank lines left out, fused_sources_sha256) is
# TRAFFIC_SOURCES_SHA256: any other hash reports the traffic as null.
# 212,900 voxels: 349.6 MB read and 35.4 MB written in one launch (profiles/k_iter_fused_hcp_brain_dram_traffic.md).
TRAFFIC_BYTES_PER_VOXEL_ITER = 1808.1
TRAFFIC_SOURCES_SHA256 = "b5f4be7847b910ed176cbdcea53adf8ad0972a350ff87f05f534bf71c9508761"
FUSED_SOURCES = ("prism_kernels.cuh", "prism_device.cuh", "prism_kset.cuh", "bessel_fit.h", "prism_k3.cu")
# FP32 lanes per SM on GB300 (4 sub-partitions x 32); the peak multiplies them by the device's
# SM count, 2 flops per fused multiply-add and the maximum SM clock seen by nvidia-smi.
FP32_LANES_PER_SM = 128


def flops_per_measurement(loss, cal, K, shell):
    """FP32 flops (fused multiply-add = 2) per (voxel, measurement) pair of the fused kernel's
    loop, counted from its algorithm. Per-measurement loop, MSE: the 17 + 28 K above. With
    calibration add 11: e^alpha_n B, S0 T, y_hat = . S + beta_n (4), the masked residual (3),
    q = r e^alpha B, q S and its running sum (3), the alpha / beta partials' reduce-scatter (1
    per value and measurement on average, 6 adds per 4 measurements and value) -- 28 + 28 K.
    Rician NLL (Eq. 9), without calibration: the MSE's residual and square (4) give way to
    y_hat = S0 T (1) and the NLL terms (71: z = y |y_hat| / sigma^2 2; Q(z) and L(z) from the
    fitted functions of 4/z, 55 -- two degree-12 Horner chains 48, the argument and scale 3,
    log terms 4; (y - |y_hat|)^2, y |y_hat| Q and L sums 9; dL/dy_hat 4; the rest 1) -- 85 + 28 K;
    with calibration 94 + 28 K; the count keeps the two degree-12 chains of the earlier two-branch
    evaluation (the segment tables' degree-7 chains take 20 fewer). Shell loop: 4 + 26 K (see
    FLOPS_PER_PAIR_SHELL); with the Rician NLL the residual and its square (3) give way to the NLL
    terms (50: z 2, segment and argument 4, the degree-7 chains 28, Q and L 3, (y - |y_hat|)^2, y |y_hat| Q
    and L sums 9, dL/dy_hat 4); calibration adds e^alpha_n B 1, y_hat 2, q 1, u and its sum 2, the partials'
    reduce-scatter 1, and the residual's 1 with the MSE."""
    if shell:
        return 4 + 26 * K + (47 if loss == "nll" else 0) + (0 if not cal else 7 if loss == "nll" else 8)
    if loss == "mse":
        return (28 + 28 * K) if cal else (17 + 28 * K)
    return (94 + 28 * K) if cal else (85 + 28 * K)


def flops_per_voxel_iteration(bvals, loss, cal, K, shell):
    """Per voxel of one volume: b = 0 measurements cost FLOPS_PER_B0_PAIR(_SHELL) where the loop
    takes them apart (MSE without calibration: the shell loop's b = 0 shell, or the leading b = 0
    pairs of the per-measurement loop); every other measurement the loop's full cost."""
    bv = np.asarray(bvals)
    n0 = int(np.count_nonzero(bv == 0))
    if loss == "mse" and not cal:
        nb0 = n0 if shell else 2 * (n0 // 2)
    else:
        nb0 = 0
    per_b0 = FLOPS_PER_B0_PAIR_SHELL if shell else FLOPS_PER_B0_PAIR
    return (len(bv) - nb0) * flops_per_measurement(loss, cal, K, shell) + nb0 * per_b0


def fp32_peak_tflops(device_index=0):
    """SMs x 128 FP32 lanes x 2 flops x the maximum SM clock nvidia-smi reports (2070 MHz if
    it reports none)."""
    import torch
    n_sm = torch.cuda.get_device_properties(device_index).multi_processor_count
    mhz = 2070.0
    try:
        out = subprocess.run(["nvidia-smi", "-i", str(device_index), "--query-gpu=clocks.max.sm",
                              "--format=csv,noheader,nounits"], capture_output=True, text=True, timeout=20).stdout
        mhz = float(out.strip().splitlines()[0])
    except (OSError, ValueError, IndexError, subprocess.SubprocessError):
        pass
    return n_sm * FP32_LANES_PER_SM * 2 * mhz * 1e6 / 1e12, f"{n_sm} SMs x {FP32_LANES_PER_SM} x 2 x {mhz:.0f} MHz"


def kernel_name(shape):
    """The iteration kernel of a Fitter with this shape()."""
    return "k_iter_local" if shape["iterations_per_launch"] > 1 else "k_iter_fused"


def speed_leg(vols, kw, steps, warmup, unfused_steps=2):
    """Fused iterations (as step() runs them, CUDA events), the iteration kernel's roofline fraction from
    the timing pass of profile(), and the plain per-patch path on the same volumes. `vols` hold device
    signals."""
    import torch
    import paper_2604_00250_gb300 as prism
    f = prism.Fitter(vols, prism.options(**kw))
    f.step(warmup)
    f.sync()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    f.step(steps)
    e1.record()
    f.sync()
    ms = e0.elapsed_time(e1) / steps
    prof = f.profile(20)
    shape = f.shape()
    K = int(kw.get("K", 3))
    loss, cal = kw.get("loss", "mse"), bool(kw.get("calibration", False))
    flops = sum(int(np.count_nonzero(v.mask)) * flops_per_voxel_iteration(v.bvals, loss, cal, K, shape["shell_loop"])
                for v in vols)
    peak, peak_src = fp32_peak_tflops()
    achieved = flops / (prof["fused_ms"] / 1e3) / 1e12
    V = f.n_vox
    f.close()
    out = {"value": V / (ms / 1e3), "ms_per_step": ms, "steps": steps, "profile_ms": prof, "launch": shape,
           "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                        "kernel": kernel_name(shape), "flops_per_iteration": flops, "peak_source": "derived: " + peak_src}}
    if unfused_steps:
        fu = prism.Fitter(vols, prism.options(**dict(kw, fused=0, use_graph=0)))
        fu.step(1)
        fu.sync()
        u0, u1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        u0.record()
        fu.step(unfused_steps)
        u1.record()
        fu.sync()
        ms_u = u0.elapsed_time(u1) / unfused_steps
        fu.close()
        out["unfused"] = {"value": V / (ms_u / 1e3), "ms_per_step": ms_u, "steps": unfused_steps}
        out["speedup_vs_unfused"] = ms_u / ms
    return out


def strip_c_comments(src):
    """C/C++ source without its comments and blank lines (string and character literals kept
    whole), so that a change of comments alone leaves the fused-kernel hash as it was."""
    out, i, n = [], 0, len(src)
    while i < n:
        c = src[i]
        if c in "\"'":
            j = i + 1
            while j < n and src[j] != c:
                j += 2 if src[j] == "\\" else 1
            out.append(src[i:j + 1])
            i = j + 1
        elif src.startswith("//", i):
            j = src.find("\n", i)
            i = n if j < 0 else j
        elif src.startswith("/*", i):
            j = src.find("*/", i + 2)
            i = n if j < 0 else j + 2
        else:
            out.append(c)
            i += 1
    lines = (ln.rstrip() for ln in "".join(out).split("\n"))
    return "\n".join(ln for ln in lines if ln)


def fused_sources_sha256():
    """SHA-256 of the fused kernel's sources, comments and blank lines left out."""
    import hashlib
    h = hashlib.sha256()
    for name in FUSED_SOURCES:
        with open(os.path.join(ROOT, "paper_2604_00250_gb300", "csrc", name), encoding="utf-8") as fh:
            h.update(strip_c_comments(fh.read()).encode("utf-8"))
    return h.hexdigest()


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def cfg_dict(V, extra=None):
    d = {"workload": WORKLOAD, "voxels": int(V), "n_meas": 288, "K": K_FIB, "loss": "mse", "patch_dim": 16,
         "priors": "repulsion+sparsity+huber_laplacian+directional_continuity",
         "l2": "inputs larger than L2: 854 MB packed signal read every step"}
    if extra:
        d.update(extra)
    return d


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled every 200 ms while active."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
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
        rows = []
        for line in open(self.path):
            p = [x.strip() for x in line.split(",")]
            if len(p) >= 9:
                rows.append(p)
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no sample"], "samples": 0}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower().startswith("active")})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def make_brain(seed, device, scale=1.0):
    import phantoms as P
    if scale == 1.0:
        return P.brain_phantom(seed=seed, device=device)
    shape = tuple(int(round(s * scale)) for s in (145, 174, 145))
    semi = tuple(a * scale for a in (52.8, 63.4, 52.8))
    return P.brain_phantom(seed=seed, device=device, shape=shape, semi=semi)


def patch_sample(vol, n_patches, patch_dim=16):
    """Ids of the n fullest 16^3 patches (a bounded, deterministic sample of the volume)."""
    mask = vol.mask.astype(bool)
    coords = np.argwhere(mask)
    pshape = tuple(-(-s // patch_dim) for s in mask.shape)
    pid = np.ravel_multi_index(tuple((coords // patch_dim).T), pshape)
    ids, counts = np.unique(pid, return_counts=True)
    order = np.argsort(-counts, kind="stable")
    return ids[order[:n_patches]], int(counts[order[:n_patches]].sum())


def oracle_rate(vol, n_patches, iters, warm=1):
    """Oracle voxel-iterations/s on whole patches of the workload (host cores)."""
    import torch
    import phantoms as P
    from oracle import prism_oracle as O
    ids, nvox = patch_sample(vol, n_patches)
    o = O.Options(K=K_FIB, loss="mse", patch_dim=16, **PRIORS)
    ov = O.OracleVolume(vol.mask, vol.signal, vol.bvals, vol.bvecs, o, patches=ids)
    th = torch.as_tensor(P.default_init(ov.n_vox, K_FIB, 0)).double()
    gp = O.group_init(ov)
    adam = O.Adam(o)
    times = []
    for it in range(warm + iters):
        t0 = time.perf_counter()
        adam.t += 1
        J, _, g, _ = O.value_and_grad(ov, th, gp, n_norm=ov.n_mask)
        th = adam.step("theta", th, g)
        times.append(time.perf_counter() - t0)
    dt = sum(times[warm:])
    return nvox * iters / dt, nvox, dt, torch.get_num_threads()


def oracle_leg(vols, kw, iters=3, max_voxels=20000):
    """The oracle as it stands on the host's cores: voxel-iterations/s of value_and_grad + Adam on
    a bounded sample -- the volumes in order, each whole or (above max_voxels) its fullest 16^3
    patches with the volume's |M|, until max_voxels."""
    import torch
    import phantoms as P
    from oracle import prism_oracle as O
    o = O.Options(**{k: v for k, v in kw.items() if hasattr(O.Options, k)})
    left, nvox, dt = max_voxels, 0, 0.0
    for v in vols:
        if left <= 0:
            break
        patches = None
        if v.n_vox > left:
            m = np.asarray(v.mask).astype(bool)
            coords = np.argwhere(m)
            pshape = tuple(-(-s // o.patch_dim) for s in m.shape)
            ids, counts = np.unique(np.ravel_multi_index(tuple((coords // o.patch_dim).T), pshape), return_counts=True)
            order = np.argsort(-counts, kind="stable")
            keep = np.cumsum(counts[order]) <= left
            keep[0] = True
            patches = ids[order][keep]
        sig = v.signal.cpu().numpy() if hasattr(v.signal, "cpu") else np.asarray(v.signal)
        ov = O.OracleVolume(v.mask, sig, v.bvals, v.bvecs, o, patches=patches)
        th = torch.as_tensor(P.default_init(ov.n_vox, o.K, 0)).double()
        gp = O.group_init(ov)
        adam = O.Adam(o)
        t0 = time.perf_counter()
        for _ in range(iters):
            adam.t += 1
            _, _, g, gg = O.value_and_grad(ov, th, gp, n_norm=ov.n_mask)
            th = adam.step("theta", th, g)
            for name, gk in gg.items():
                gp[name] = adam.step((name, 0), gp[name], gk)
        dt += time.perf_counter() - t0
        nvox += ov.n_vox
        left -= ov.n_vox
    return {"value": nvox * iters / dt, "unit": UNIT, "cores": torch.get_num_threads(), "kind": "oracle",
            "sample": f"{nvox} voxels x {iters} iterations, {dt:.1f} s"}


def run_small(args):
    """The crossing patch (8^3, N = 96, MSE, K = 3; 'patch') and the crossing sweep (16 volumes
    of 10^3 at 20-90 deg, N = 96, K = 3, MSE and the Rician NLL with sigma per volume; 'sweep'):
    fused and unfused speed, the fused kernel's roofline fraction and the oracle on the host."""
    import torch
    import phantoms as P
    if args.workload == "patch":
        cases = [("crossing_patch_8cubed_N96_K3_mse", [P.crossing_patch(args.seed)], dict(K=3, loss="mse", patch_dim=8))]
    else:
        vols = P.crossing_sweep(args.seed)
        cases = [(f"crossing_sweep_16x10cubed_N96_K3_{l}", vols, dict(K=3, loss=l, patch_dim=10)) for l in ("mse", "nll")]
    import types
    for name, vols, kw in cases:
        gv = [types.SimpleNamespace(mask=v.mask, signal=torch.as_tensor(v.signal, device="cuda"), bvals=v.bvals,
                                    bvecs=v.bvecs, init=None) for v in vols]
        leg = speed_leg(gv, kw, min(args.steps, 500), args.warmup, unfused_steps=0 if args.no_unfused else 5)
        line = {"workload": name, "voxels": int(sum(v.n_vox for v in vols)), "unit": UNIT, **leg, "options": kw}
        if not args.no_cpu:
            line["cpu_baseline"] = oracle_leg(vols, kw)
        print(json.dumps(line), flush=True)
    return 0


def run_reference(args):
    world, rank, _ = dist_env()
    if rank != 0:
        return 0
    import torch
    vol = make_brain(args.seed, "cpu", args.brain_scale)
    V = vol.n_vox
    ids, nvox = patch_sample(vol, 1)
    import phantoms as P
    from oracle import prism_oracle as O
    o = O.Options(K=K_FIB, loss="mse", patch_dim=16, **PRIORS)
    ov = O.OracleVolume(vol.mask, vol.signal, vol.bvals, vol.bvecs, o, patches=ids)
    th = torch.as_tensor(P.default_init(ov.n_vox, K_FIB, 0)).double()
    gp = O.group_init(ov)
    adam = O.Adam(o)

    def one():
        adam.t += 1
        _, _, g, _ = O.value_and_grad(ov, th, gp, n_norm=ov.n_mask)
        return adam.step("theta", th, g)

    for _ in range(args.warmup):
        th = one()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        th = one()
    dt = time.perf_counter() - t0
    value = nvox * args.steps / dt
    cores = torch.get_num_threads()
    sample = f"one 16^3 patch ({nvox} voxels) of the {V}-voxel brain per step"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
            "higher_is_better": True, "scaling": "strong", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": cfg_dict(V, {"sample": sample}),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import torch
    import torch.distributed as dist
    import types
    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    import paper_2604_00250_gb300 as prism
    from paper_2604_00250_gb300 import shard
    dev = torch.device("cuda", local)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    def max_over_ranks(x):
        if world == 1:
            return x
        t = torch.tensor([x], dtype=torch.float64, device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        return float(t.item())

    # one brain; with N > 1 ranks each fits its share of the 16^3 patches (occupancy-balanced,
    # the whole brain's |M| as the normaliser) and no data crosses ranks while fitting
    vol = make_brain(args.seed, "cuda", args.brain_scale)
    V_all = vol.n_vox
    N = vol.n_meas
    whole = types.SimpleNamespace(mask=vol.mask, signal=vol.signal, bvals=vol.bvals, bvecs=vol.bvecs, init=None,
                                  norm_count=0)
    part = shard.shard_volume(whole, 16, rank, world)[0] if world > 1 else whole
    V = int(np.count_nonzero(part.mask))
    sig_dev = torch.as_tensor(part.signal, device=dev)
    vdev = types.SimpleNamespace(mask=part.mask, signal=sig_dev, bvals=vol.bvals, bvecs=vol.bvecs, init=None,
                                 norm_count=part.norm_count)
    opts = prism.options(K=K_FIB, loss="mse", patch_dim=16, fused=1, use_graph=1, autotune=int(args.autotune),
                         threads_per_voxel=args.threads_per_voxel, **PRIORS)
    f = prism.Fitter([vdev], opts)
    stream = torch.cuda.current_stream()
    # ---- timed region: K fused iterations (graph replay), inputs resident in HBM
    f.step(args.warmup)
    f.sync()
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.25)
    barrier()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    f.step(args.steps)
    e1.record(stream)
    e1.synchronize()
    barrier()
    ck = clocks.stop()
    f.sync()
    ms_total = max_over_ranks(e0.elapsed_time(e1))
    ms_step = ms_total / args.steps
    value = V_all * args.steps / (ms_total / 1e3)
    # ---- live per-kernel timing (CUDA events around each kernel class, no graph)
    prof = f.profile(min(args.steps, 50))
    fused_ms = prof["fused_ms"]
    nb0 = 2 * (int(np.count_nonzero(np.asarray(vol.bvals) == 0)) // 2)
    shape = f.shape()
    per_pair = FLOPS_PER_PAIR_SHELL if shape["shell_loop"] else FLOPS_PER_PAIR
    per_b0 = FLOPS_PER_B0_PAIR_SHELL if shape["shell_loop"] else FLOPS_PER_B0_PAIR
    achieved = V * ((N - nb0) * per_pair + nb0 * per_b0) / (fused_ms / 1e3) / 1e12
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    sm_max_mhz = ck.get("sm_max_mhz") or 2070.0
    peak = n_sm * FP32_LANES_PER_SM * 2 * sm_max_mhz * 1e6 / 1e12
    peak_at_median = n_sm * FP32_LANES_PER_SM * 2 * ck["sm_mhz"] * 1e6 / 1e12 if ck.get("sm_mhz") else None
    ffma_measured = prism.microbench("ffma") / 1e12
    sha = fused_sources_sha256()
    traffic = (V * TRAFFIC_BYTES_PER_VOXEL_ITER
               if TRAFFIC_BYTES_PER_VOXEL_ITER and sha == TRAFFIC_SOURCES_SHA256 else None)
    loss_last = float(f.loss()[0])
    tile = f.shape()
    f.close()
    # ---- plain path: separate launches per patch and step, no graph
    unfused = None
    if not args.no_unfused:
        fu = prism.Fitter([vdev], prism.options(K=K_FIB, loss="mse", patch_dim=16, fused=0, use_graph=0, **PRIORS))
        fu.step(2)
        fu.sync()
        n_u = 5
        u0 = torch.cuda.Event(enable_timing=True)
        u1 = torch.cuda.Event(enable_timing=True)
        u0.record(stream)
        fu.step(n_u)
        u1.record(stream)
        u1.synchronize()
        fu.sync()
        ms_u = max_over_ranks(u0.elapsed_time(u1)) / n_u
        unfused = {"value": V_all / (ms_u / 1e3), "ms_per_step": ms_u, "steps": n_u,
                   "launches_per_step": None}
        fu.close()
    # ---- end to end through prism_fit with HOST buffers (copies inside the timed region)
    e2e = None
    if not args.no_e2e:
        sig_host = torch.empty(tuple(part.signal.shape), dtype=torch.float32, pin_memory=True)
        sig_host.copy_(torch.as_tensor(part.signal))
        vhost = types.SimpleNamespace(mask=part.mask, signal=sig_host, bvals=vol.bvals, bvecs=vol.bvecs, init=None,
                                      norm_count=part.norm_count)
        n_e2e = args.e2e_iters
        out = torch.empty((V, 4 * K_FIB + 5), dtype=torch.float32, pin_memory=True)
        import ctypes
        from paper_2604_00250_gb300 import _lib
        lib = _lib.load()
        keep = []
        arr, nv = prism._volumes_array([vhost], keep)
        loss_out = np.empty(1, dtype=np.float64)
        # three complete calls, the median reported, the fastest and all three listed: on the
        # shared GB300 hosts the wall time of a call varies by up to 15 % (the device time of its
        # iterations does not)
        runs = []
        for _ in range(3):
            barrier()
            t0 = time.perf_counter()
            _lib.check(lib.prism_fit(arr, nv, ctypes.byref(opts), n_e2e, ctypes.c_void_p(out.data_ptr()),
                                     loss_out.ctypes.data, prism.MEM_HOST, ctypes.c_void_p(stream.cuda_stream)))
            torch.cuda.synchronize()
            runs.append(max_over_ranks(time.perf_counter() - t0))
        dt = float(np.median(runs))
        h2d = sig_host.numel() * 4 + vol.mask.size + N * 16
        d2h = out.numel() * 4 + 8
        e2e = {"value": V_all * n_e2e / dt, "unit": UNIT, "h2d_bytes_per_step": h2d / n_e2e,
               "d2h_bytes_per_step": d2h / n_e2e, "iterations": n_e2e, "seconds": dt,
               "value_fastest": V_all * n_e2e / min(runs), "seconds_fastest": min(runs),
               "seconds_all_calls": [round(r, 4) for r in runs], "timing": "wall clock, median of 3 calls",
               "call": "prism_fit (init + iterations + readout), pinned host signal and parameters"}
    # ---- CPU baseline: the FP64 oracle on a bounded sample (rank 0, N = 1 only)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        rate, nvox, dt, cores = oracle_rate(vol, args.cpu_patches, args.cpu_iters)
        cpu = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{args.cpu_patches} fullest 16^3 patches ({nvox} voxels) x {args.cpu_iters} iterations, "
                         f"{dt:.1f} s"}
        # the same oracle on one core (one patch, five iterations)
        import torch
        nt = torch.get_num_threads()
        torch.set_num_threads(1)
        try:
            rate1, nvox1, dt1, _ = oracle_rate(vol, 1, 5)
        finally:
            torch.set_num_threads(nt)
        cpu["value_1core"] = rate1
        cpu["sample_1core"] = f"1 fullest 16^3 patch ({nvox1} voxels) x 5 iterations, {dt1:.1f} s"
    # per iteration: the Huber-Laplacian preparation, the neighbour-prior rows and the fused
    # kernel (groups finalised inside it)
    launches = 1 + (1 if PRIORS["lam_sp"] > 0 else 0) + (1 if (PRIORS["lam_sp"] > 0 or PRIORS["lam_dir"] > 0) else 0)
    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "strong",
                "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": cfg_dict(V_all, {"timing": "CUDA events, graph replay, max over ranks",
                                           "partition": (f"{world} ranks, 16^3 patches balanced by voxel count, "
                                                         f"rank 0 fits {V} voxels" if world > 1 else "one GPU"),
                                       "brain_scale": args.brain_scale, "launch": tile}),
                "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                             "frac": achieved / peak, "traffic": traffic,
                             "flops_per_voxel_iteration": (N - nb0) * per_pair + nb0 * per_b0,
                             "traffic_unit": "bytes per launch (ncu dram read + write, scaled capture)",
                             "kernel": "k_iter_fused", "kernel_ms": fused_ms,
                             "peak_source": f"derived: {n_sm} SMs x {FP32_LANES_PER_SM} FP32 lanes x 2 x "
                                            f"{sm_max_mhz:.0f} MHz (maximum SM clock sampled)",
                             "peak_at_median_clock": peak_at_median,
                             "ffma_microbench": ffma_measured,
                             "frac_of_ffma_microbench": achieved / ffma_measured,
                             "fused_sources_sha256": sha},
                "unfused": unfused,
                "speedup_vs_unfused": (value / unfused["value"]) if unfused else None,
                "profile_ms": prof, "final_loss": loss_last,
                "clocks": ck, "e2e": e2e, "cpu_baseline": cpu,
                "gpu_launches": launches * args.steps}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


# Crossing-fiber benchmark configuration (Sec. 3 "Configuration": K = 2, MSE and NLL with
# learned sigma, direction repulsion only, no spatial priors); 300 Adam iterations.
CROSS_OPTS = dict(K=2, lam_rep=0.01, lam_sparse=0.0, lam_sp=0.0, lam_dir=0.0, patch_dim=16)


def run_calibrated(args):
    """Speed of the calibrated Rician-NLL configurations (one JSON line each, not the headline):
    'bundle' = the 64^3 bundle phantom (N = 360, bias field and per-measurement affine, SNR 20);
    'multi' = the batch of 12 volumes of edge 32..128 (schemes of 96/288/360 measurements,
    about 4 M voxels), both with K = 3, NLL with learned sigma, full calibration and the
    neighbour priors, in 16^3 patches. Reports voxel-iterations/s of graph-replayed fused
    iterations, the per-kernel times and the device memory the fit holds."""
    import types
    import torch
    import phantoms as P
    import paper_2604_00250_gb300 as prism
    vols = ([P.bundle_phantom(args.seed, device="cuda")] if args.workload == "bundle"
            else P.multi_volume_batch(args.seed, device="cuda"))
    gv = [types.SimpleNamespace(mask=v.mask, signal=torch.as_tensor(v.signal, device="cuda"), bvals=v.bvals,
                                bvecs=v.bvecs, init=None) for v in vols]
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    opts = dict(K=3, loss="nll", calibration=True, lam_sp=0.01, lam_dir=0.005, patch_dim=16)
    f = prism.Fitter(gv, prism.options(**opts))
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0]
    n_vox, n_groups = f.n_vox, f.n_groups
    f.close()
    leg = speed_leg(gv, opts, min(args.steps, 500), args.warmup, unfused_steps=0 if args.no_unfused else 2)
    line = {"workload": ("bundle_64cubed_N360_nll_calibrated" if args.workload == "bundle"
                         else "multi_volume_12_edges_32_to_128_N96_288_360_nll_calibrated"),
            "voxels": n_vox, "volumes": n_groups, "unit": "voxel-iterations/s", **leg,
            "signal_bytes": int(sum(v.signal.numel() * 4 for v in gv)), "fit_device_bytes": int(held),
            "options": opts}
    if not args.no_cpu:
        line["cpu_baseline"] = oracle_leg(vols, opts)
    print(json.dumps(line), flush=True)
    return 0


def run_slabs(args):
    """The paper's whole-brain pipeline (Sec. 3 "Configuration"): the HCP-shaped brain cut into
    30-slice slabs with a 5-slice overlap, K = 3, MSE with the full prior suite, Rprop (the
    paper's solver), 100 iterations per slab, then the stitched whole-volume maps. All slabs are one batch. Times the whole job
    from pinned host buffers (set-up, iterations, stitch, read-out) with the wall clock."""
    import types
    import torch
    import paper_2604_00250_gb300 as prism
    vol = make_brain(args.seed, "cuda")
    sig_host = torch.empty(vol.signal.shape, dtype=torch.float32, pin_memory=True)
    sig_host.copy_(torch.as_tensor(vol.signal))
    vh = types.SimpleNamespace(mask=vol.mask, signal=sig_host, bvals=vol.bvals, bvecs=vol.bvecs, init=None)
    opts = prism.options(K=K_FIB, loss="mse", patch_dim=16, lam_orphan=0.01, lam_order=0.01, optimizer="rprop",
                         **PRIORS)
    iters = 100
    # the stitched maps go into pinned host arrays allocated once, like the input signal
    V_all = vol.n_vox
    outs = tuple(torch.empty(s, dtype=torch.float32, pin_memory=True)
                 for s in ((V_all,), (V_all, K_FIB + 3), (V_all,), (V_all, K_FIB, 3)))
    times = []
    for rep in range(2):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f = prism.Fitter(vh, opts, slabs=(30, 5))
        f.step(iters)
        s0, fr, fin, d = f.stitch(out=outs)
        torch.cuda.synchronize()
        times.append(time.perf_counter() - t0)
        n_slab_vox, n_slabs = f.n_vox, f.n_groups
        f.close()
    dt = min(times)
    # the fused kernel's roofline fraction on the slab batch, and the plain per-patch path
    f = prism.Fitter(vh, opts, slabs=(30, 5))
    f.step(3)
    prof = f.profile(20)
    shape = f.shape()
    f.close()
    flops = n_slab_vox * flops_per_voxel_iteration(vol.bvals, "mse", False, K_FIB, shape["shell_loop"])
    peak, peak_src = fp32_peak_tflops()
    achieved = flops / (prof["fused_ms"] / 1e3) / 1e12
    unfused = None
    if not args.no_unfused:
        plain = prism.options(K=K_FIB, loss="mse", patch_dim=16, lam_orphan=0.01, lam_order=0.01, optimizer="rprop",
                              fused=0, use_graph=0, **PRIORS)
        fu = prism.Fitter(vh, plain, slabs=(30, 5))
        fu.step(1)
        fu.sync()
        u0, u1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        u0.record()
        fu.step(2)
        u1.record()
        fu.sync()
        ms_u = u0.elapsed_time(u1) / 2
        fu.close()
        unfused = {"value": n_slab_vox / (ms_u / 1e3), "ms_per_step": ms_u, "steps": 2,
                   "unit": "slab voxel-iterations/s"}
    line = {"workload": "hcp_shaped_brain_slabs_30_overlap_5_K3_mse_full_priors_rprop_100_iterations",
            "voxels": int(s0.shape[0]), "slabs": n_slabs, "slab_voxels": n_slab_vox, "iterations": iters,
            "seconds": dt, "value": n_slab_vox * iters / dt, "unit": "slab voxel-iterations/s",
            "timing": "wall clock, pinned host signal, set-up + iterations + stitch + read-out, best of 2",
            "profile_ms": prof, "launch": shape,
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                         "kernel": "k_iter_fused", "peak_source": "derived: " + peak_src},
            "unfused": unfused,
            "speedup_vs_unfused": (unfused["ms_per_step"] / (prof["iter_ms"])) if unfused else None,
            "paper_context": "the paper reports about 12 minutes for this pipeline on an RTX A6000"}
    print(json.dumps(line), flush=True)
    return 0


def run_disco(args):
    """The DiSCo1-shaped fit (Sec. 3 "Datasets" / "Configuration"): a 40^3 phantom of curved
    bundles, 4 shells with b up to 13,192 s/mm^2 (4 b = 0 + 90 directions at 1000 / 3000 / 7000 /
    13,192, N = 364), SNR 50, K = 5, Rician NLL with learned sigma, the topology and spatial
    priors of Sec. 2.4, 300 iterations. Wall-clock time of the whole fit from pinned host
    buffers."""
    import types
    import torch
    import phantoms as P
    import paper_2604_00250_gb300 as prism
    sch = P.make_scheme(4, [(1000, 90), (3000, 90), (7000, 90), (13192, 90)], args.seed)
    vol = P.bundle_phantom(args.seed, edge=40, snr=50.0, scheme=sch, device="cuda")
    sig_host = torch.empty(tuple(vol.signal.shape), dtype=torch.float32, pin_memory=True)
    sig_host.copy_(torch.as_tensor(vol.signal))
    vh = types.SimpleNamespace(mask=vol.mask, signal=sig_host, bvals=vol.bvals, bvecs=vol.bvecs, init=None)
    # the topology priors (repulsion, sparsity, orphan-WM, directional continuity, ordering)
    # and the Huber-Laplacian smoothness, at the weights of Sec. 2.4
    opts = prism.options(K=5, loss="nll", patch_dim=16, lam_orphan=0.01, lam_order=0.01, **PRIORS)
    iters = 300
    times = []
    for rep in range(2):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f = prism.Fitter(vh, opts)
        f.step(iters)
        th = f.params_host()
        torch.cuda.synchronize()
        times.append(time.perf_counter() - t0)
        prof = f.profile(20)
        V = f.n_vox
        f.close()
    dt = min(times)
    vdev = types.SimpleNamespace(mask=vol.mask, signal=torch.as_tensor(vol.signal, device="cuda"), bvals=vol.bvals,
                                 bvecs=vol.bvecs, init=None)
    leg = speed_leg([vdev], dict(K=5, loss="nll", patch_dim=16, lam_orphan=0.01, lam_order=0.01, **PRIORS), 100, 5,
                    unfused_steps=0 if args.no_unfused else 2)
    line = {"workload": "disco1_shaped_40cubed_N364_K5_nll_priors_300_iterations", "voxels": V, "iterations": iters,
            "seconds": dt, "value": V * iters / dt, "unit": "voxel-iterations/s", "profile_ms": prof,
            "timing": "wall clock, pinned host signal, set-up + iterations + read-out, best of 2",
            "graph_replay": {k: leg[k] for k in ("value", "ms_per_step", "launch", "roofline")},
            "unfused": leg.get("unfused"), "speedup_vs_unfused": leg.get("speedup_vs_unfused")}
    print(json.dumps(line), flush=True)
    return 0


def run_crossing(args):
    """Quality of the fit on the crossing-fiber benchmark layout (16 angles + single-fiber
    controls, N = 193) at each SNR and both data terms: one JSON line per run with the
    best-match angular error per angle, overall, recall and F1 (Sec. 3 "Tracking & metrics";
    peaks are fibers with at least 15 % of the white-matter fraction)."""
    import torch
    import phantoms as P
    import paper_2604_00250_gb300 as prism
    from paper_2604_00250_gb300 import crossing
    for snr in args.cross_snr:
        vol = P.crossing_benchmark(snr=snr, seed=args.seed, n_per_case=args.cross_voxels)
        for loss in ("mse", "nll"):
            f = prism.Fitter(vol, prism.options(loss=loss, **CROSS_OPTS))
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            f.step(args.cross_iters)
            e1.record()
            f.sync()
            d, _, pk = f.fibers(0.15)
            per, overall, rec, prec, f1 = crossing.score(d, pk, vol.gt["dirs"], vol.gt["ffib"], vol.gt["case"])
            final_loss = float(f.loss()[0])
            prof = f.profile(10)
            shape = f.shape()
            flops = f.n_vox * flops_per_voxel_iteration(vol.bvals, loss, False, CROSS_OPTS["K"], shape["shell_loop"])
            peak, _ = fp32_peak_tflops()
            roof = {"bound": "alu", "achieved": flops / (prof["fused_ms"] / 1e3) / 1e12, "peak": peak,
                    "unit": "TFLOP/s", "kernel": kernel_name(shape)}
            roof["frac"] = roof["achieved"] / peak
            fu = prism.Fitter(vol, prism.options(loss=loss, fused=0, use_graph=0, **CROSS_OPTS))
            fu.step(1)
            fu.sync()
            u0, u1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            u0.record()
            fu.step(5)
            u1.record()
            fu.sync()
            unfused_ms = u0.elapsed_time(u1) / 5
            fu.close()
            line = {"workload": "crossing_benchmark_N193_K2", "snr": snr, "loss": loss, "voxels": f.n_vox,
                    "iterations": args.cross_iters, "fit_ms": e0.elapsed_time(e1),
                    "single_fiber_deg": per[0],
                    "per_angle_deg": {str(a): per[i + 1] for i, a in enumerate(P.BENCH_ANGLES)},
                    "overall_deg": overall, "recall": rec, "precision": prec, "f1": f1,
                    "final_loss": final_loss, "profile_ms": prof, "launch": shape, "roofline": roof,
                    "unfused_ms_per_step": unfused_ms, "speedup_vs_unfused": unfused_ms / prof["iter_ms"]}
            print(json.dumps(line), flush=True)
            f.close()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--autotune", action="store_true")
    ap.add_argument("--brain-scale", type=float, default=1.0,
                    help="scale the brain grid (profiling of smaller cases; 1.0 = the benchmark workload)")
    ap.add_argument("--threads-per-voxel", type=int, default=0, choices=[0, 1, 4, 16],
                    help="force the fused kernel's lanes per voxel (0 = chosen from the voxel count)")
    ap.add_argument("--e2e-iters", type=int, default=500)
    ap.add_argument("--cpu-patches", type=int, default=4)
    ap.add_argument("--cpu-iters", type=int, default=20)
    ap.add_argument("--no-unfused", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--workload", default="brain",
                    choices=["brain", "crossing", "bundle", "multi", "slabs", "disco", "patch", "sweep"],
                    help="crossing: fit quality on the crossing-fiber benchmark layout; patch / sweep: speed "
                         "on the 8^3 crossing patch and the 16-volume crossing sweep; bundle / multi: speed "
                         "of the calibrated NLL configurations; slabs: the whole-brain slab pipeline; "
                         "disco: the DiSCo1-shaped K = 5 NLL fit (none of these is the headline)")
    ap.add_argument("--cross-snr", type=float, nargs="+", default=[10.0, 30.0, 50.0])
    ap.add_argument("--cross-voxels", type=int, default=200, help="voxels per angle (and single-fiber controls)")
    ap.add_argument("--cross-iters", type=int, default=300)
    args = ap.parse_args()
    if args.workload == "crossing":
        return run_crossing(args)
    if args.workload in ("bundle", "multi"):
        return run_calibrated(args)
    if args.workload in ("patch", "sweep"):
        if args.warmup < 3:
            args.warmup = 3
        return run_small(args)
    if args.workload == "slabs":
        return run_slabs(args)
    if args.workload == "disco":
        return run_disco(args)
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
