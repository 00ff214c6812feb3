#!/usr/bin/env python3
"""Throughput of the RenderMap pose-cost hot path on one GB300 (or N, one replica each).

One step = the whole hot path for one batch: render the labelled 1M-triangle map's z-buffer
from each of 256 candidate poses at 640x480, apply Table I per pixel with the truncated
least-squares residual, and reduce the adjoint gradient and Gauss-Newton matrix per pose
(rm_cost_grad). Metric: pose evaluations per second. Prints ONE JSON line on rank 0.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
  python bench.py --workload tracking     # 64 mixed-sensor agents, rm_align_batch per frame
  python bench.py --workload icp          # point-to-plane ICP terms and alignments (Sec. V)
  python bench.py --workload normals      # Eq. 2 normals of 64 depth images per step
  python bench.py --workload vgrad        # vertex-position gradient of 16 poses per step
  python bench.py --workload lidar        # 64 poses, 1024x64 Lidar, 2M-triangle terrain; LM
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "pose evals/s (render+residual+grad) 640x480, 1M tris; % of HBM roofline"
UNIT = "pose evals/s"
PEAKS_FALLBACK = {"hbm_gbs": 6800.0}


def args_():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--poses", type=int, default=256)
    ap.add_argument("--seed", type=int, default=3000)
    ap.add_argument("--cpu-sample", type=int, default=64, help="poses per step of the reference arm")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--tile", default=None, help="WxH screen tile (e.g. 64x32): skip the autotuner")
    ap.add_argument("--workload", choices=["headline", "tracking", "icp", "normals", "vgrad", "lidar"],
                    default="headline")
    ap.add_argument("--frames", type=int, default=200, help="tracking: frames of the trajectory")
    ap.add_argument("--agents", type=int, default=64, help="tracking: agents (scans per frame)")
    ap.add_argument("--triangles", type=int, default=2_000_000, help="tracking: map size")
    ap.add_argument("--method", choices=["lm", "icp"], default="lm",
                    help="tracking: LM on the Table I surrogate, or point-to-plane ICP (Sec. V)")
    return ap.parse_args()


# ---- multi-rank plumbing (one process per GPU; each rank evaluates its own batch of poses, so
# the data path has no collective; only the timing is reduced, max over ranks)

def rank_info():
    """(world, rank, local rank) from the launcher's environment (1, 0, 0 without one)."""
    return (int(os.environ.get("WORLD_SIZE", "1")), int(os.environ.get("RANK", "0")),
            int(os.environ.get("LOCAL_RANK", "0")))


def rank_seed(seed, rank):
    """Each rank's synthetic batch: the same workload shape, its own candidate poses and scan."""
    return seed + 17 * rank


def max_over_ranks(x, world, device):
    """The largest of every rank's x (a time): all ranks wait for the slowest."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    if world > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_rate(world, units_per_rank, seconds):
    """Whole-job throughput: the units all ranks processed over the slowest rank's time."""
    return world * units_per_rank / seconds


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            p = json.load(fh)
        return p, "measured"
    except OSError:
        return PEAKS_FALLBACK, "fallback"


def kernel_source_hash():
    """First 16 hex digits of sha256 over the kernel sources (as recorded in profiles/)."""
    import hashlib
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_1702_06813_gb300", "csrc")
    for f in ("rm_kernels.cu", "rm_internal.cuh"):
        with open(os.path.join(csrc, f), "rb") as fh:
            h.update(hashlib.sha256(fh.read()).hexdigest().encode() + b"  " + f"paper_1702_06813_gb300/csrc/{f}\n".encode())
    return h.hexdigest()[:16]


def measured_traffic(kernel, poses_per_launch, n_tris):
    """DRAM bytes per launch of `kernel` from the ncu summary in profiles/, scaled by poses per
    launch; None when the summary is missing or was taken on different kernel sources or a
    different map."""
    path = os.path.join(ROOT, "profiles", f"{kernel}_room1M_640x480.md")
    try:
        text = open(path).read()
    except OSError:
        return None
    fields = dict(line.split(":", 1) for line in text.splitlines() if ":" in line and " " not in line.split(":", 1)[0])
    try:
        if fields["kernel_source_sha256_16"].strip() != kernel_source_hash():
            return None
        if int(fields["map_triangles"]) != int(n_tris):
            return None
        return int(fields["dram_bytes_per_launch"]) / int(fields["poses_per_launch"]) * poses_per_launch
    except (KeyError, ValueError):
        return None


def algorithmic_bytes(V, T, P):
    """Bytes one pose evaluation must touch: vertices 12 V, faces + labels 13 T, scan 5 P."""
    return {"k_cull": 0, "k_setup": 12 * V + 13 * T, "k_raster": 5 * P, "k_reduce": 0,
            "total": 12 * V + 13 * T + 5 * P}


def step_algorithmic_bytes(V, T, P, n_poses, wave_poses):
    """Bytes one batched step must move from HBM: the map once per wave of poses (every pose
    of a wave shares it) and the scan comparison once per pose."""
    waves = -(-n_poses // max(1, wave_poses))
    return (12 * V + 13 * T) * waves + 5 * P * n_poses


class Clocks:
    """nvidia-smi clock / throttle sampling while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid):
        self.uuid = uuid
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"] + (["-i", self.uuid] if self.uuid else []),
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": sorted(reasons),
                "samples": len(sm)}


def cpu_baseline(w, min_seconds=1.5):
    """The oracle as it stands on the host cores (OpenMP over poses): whole passes over the
    candidate-pose batch until at least min_seconds of wall time (about 20 core-seconds on
    a 16-core host)."""
    import oracle
    oracle.build()
    om = oracle.OracleMap(w["mesh"].vertices, w["mesh"].faces, w["mesh"].labels)
    sd, sc = w["scan"]
    poses = w["poses"]
    om.cost_batch(poses[:1], w["cam"], sd, sc)  # page in
    done, threads = 0, 1
    t0 = time.perf_counter()
    while time.perf_counter() - t0 < min_seconds:
        threads = om.cost_batch(poses, w["cam"], sd, sc)["threads"]
        done += len(poses)
    dt = time.perf_counter() - t0
    return {"value": done / dt, "unit": UNIT, "cores": int(threads), "kind": "oracle",
            "sample": f"{done // len(poses)} pass(es) over the {len(poses)} candidate poses, each a full "
                      f"640x480 render + Table I + FP64 gradient, OpenMP over poses, {dt:.1f} s wall"}


def oracle_single_thread(w, n=4):
    """The oracle as it stands on one host thread, one pose at a time (the plain CPU form):
    evaluations per second over the first n candidate poses."""
    import oracle
    oracle.build()
    om = oracle.OracleMap(w["mesh"].vertices, w["mesh"].faces, w["mesh"].labels)
    sd, sc = w["scan"]
    om.cost(w["poses"][0], w["cam"], sd, sc)  # page in
    t0 = time.perf_counter()
    for P in w["poses"][:n]:
        om.cost(P, w["cam"], sd, sc)
    return n / (time.perf_counter() - t0)


def run_reference(a):
    """The oracle timed as it stands on the host cores (OpenMP over poses), on the same
    workload, batch, metric and step count as the GPU arm (rank 0 only): each step is one
    pass over the candidate-pose batch (about 0.3 s on 16 cores for 256 poses)."""
    rank = rank_info()[1]
    if rank != 0:
        return
    import synth
    w = synth.workload_headline(a.seed, a.poses)
    import oracle
    oracle.build()
    om = oracle.OracleMap(w["mesh"].vertices, w["mesh"].faces, w["mesh"].labels)
    sd, sc = w["scan"]
    poses = w["poses"]
    for k in range(max(1, a.warmup)):
        om.cost_batch(poses, w["cam"], sd, sc)
    t0 = time.perf_counter()
    threads = 1
    for k in range(a.steps):
        threads = om.cost_batch(poses, w["cam"], sd, sc)["threads"]
    dt = time.perf_counter() - t0
    v = a.steps * len(poses) / dt
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": a.gpus,
        "steps": a.steps, "warmup": max(1, a.warmup), "ms_per_step": 1e3 * dt / a.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": w["name"], "poses_per_gpu": len(poses), "triangles": w["mesh"].n_tris,
                   "image": [w["cam"].width, w["cam"].height]},
        "cpu_baseline": {"value": v, "unit": UNIT, "cores": int(threads), "kind": "oracle",
                         "sample": f"{a.steps} passes over the {len(poses)}-pose batch, OpenMP over poses"},
        "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}))


def run_tracking(a):
    """64 agents with mixed sensors track their own trajectories over one map; every frame is
    one rm_align_batch call (5 LM iterations each, all agents in step on the device, as one
    captured graph). Observed scans are the map's free-occupied faces rendered at the true poses with
    this library's z-buffer, plus sensor noise, made outside the timed region."""
    import torch
    import paper_1702_06813_gb300 as rm
    import synth
    import __graft_entry__
    __graft_entry__.build_library()
    frac = a.triangles / 2_000_000
    w = synth.workload_tracking(a.seed + 2000, n_agents=a.agents, n_frames=a.frames,
                                target_fo=int(1_400_000 * frac), target_fu=int(600_000 * frac),
                                n_panels=max(40, int(400 * frac)))
    mesh, cams, kinds, truth = w["mesh"], w["cams"], w["kinds"], w["poses"]
    torch.cuda.set_device(0)
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    fo = mesh.labels == 0
    g_fo = rm.Map(mesh.vertices, mesh.faces[fo], mesh.labels[fo])
    intr = [rm.Intrinsics.from_camera(c) for c in cams]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(a.seed)
    n_agents = truth.shape[1]
    groups = [np.nonzero(kinds == k)[0] for k in range(3)]

    def scans_for(f):
        out = [None] * n_agents
        for k, idx in enumerate(groups):
            d = rm.render_depth(g_fo, truth[f, idx], intr[k], want_id=False)["depth"]
            sig = torch.full_like(d, 0.02) if cams[k].model != "pinhole" else 0.005 * torch.nan_to_num(d, nan=0.0)
            d = d + sig * torch.randn(d.shape, device="cuda", generator=gen)
            far = ~(d <= cams[k].range_max)
            cls = torch.where(far, torch.ones_like(d, dtype=torch.uint8), torch.zeros_like(d, dtype=torch.uint8))
            d = torch.where(far, torch.full_like(d, cams[k].range_max), d)
            for j, ag in enumerate(idx):
                out[ag] = rm.Scan(intr[k], d[j].contiguous(), cls[j].contiguous())
        return out

    rng = np.random.Generator(np.random.PCG64(a.seed + 7))
    est = np.stack([synth.perturb_fixed(truth[0, i], rng, 0.10, 1.0) for i in range(n_agents)])
    prev = est.copy()
    scans0 = scans_for(0)
    def step_batch(pairs):
        if a.method == "icp":
            return rm.icp_align_batch(gm, pairs, tol=0.3, max_iters=5, step_tol=1e-4)
        return rm.align_batch(gm, pairs, max_iters=5)

    step_batch([(scans0[i], est[i]) for i in range(n_agents)])  # warm
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    total_ms, evals = 0.0, 0
    errs = []
    for f in range(a.frames):
        scans = scans_for(f)
        if f == 0:
            init = est
        else:
            init = np.stack([est[i] @ np.linalg.inv(prev[i]) @ est[i] for i in range(n_agents)])
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        out, reps, _ = step_batch([(scans[i], init[i]) for i in range(n_agents)])
        e1.record(stream)
        torch.cuda.synchronize()
        total_ms += e0.elapsed_time(e1)
        evals += sum(1 + r["iters"] if a.method == "lm" else min(5, r["iters"] + 1) for r in reps)
        prev, est = est, out
        errs.append(np.linalg.norm(est[:, :3, 3] - truth[f, :, :3, 3], axis=1))
    value = n_agents * a.frames / (total_ms * 1e-3)
    # plain per-pose form on the first frames: one rm_align call per agent
    n_plain = min(a.frames, 5)
    plain_ms = 0.0
    for f in range(n_plain):
        scans = scans_for(f)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for i in range(n_agents):
            if a.method == "icp":
                rm.icp_align(gm, scans[i], truth[f, i], tol=0.3, max_iters=5, step_tol=1e-4)
            else:
                rm.align(gm, scans[i], truth[f, i], max_iters=5)
        torch.cuda.synchronize()
        plain_ms += (time.perf_counter() - t0) * 1e3
    plain_value = n_agents * n_plain / (plain_ms * 1e-3)
    errs = np.array(errs)
    # roofline of a frame's one batch call: algorithmic bytes per
    # call = the map once plus the scan comparison of every evaluation of every agent
    pk, pk_kind = peaks()
    p_img = [c.width * c.height for c in cams]
    evals_per_agent = 1 + 5 if a.method == "lm" else 5
    launch_bytes = 12 * mesh.n_verts + 13 * mesh.n_tris + sum(5 * p_img[k] * evals_per_agent for k in kinds)
    achieved = launch_bytes / (total_ms / a.frames * 1e-3) / 1e9
    roofline = {"bound": "hbm", "kernel": "batch graph", "achieved": achieved, "peak": pk["hbm_gbs"],
                "unit": "GB/s", "frac": achieved / pk["hbm_gbs"], "traffic": None, "peak_kind": pk_kind,
                "avg_launch_ms": total_ms / a.frames, "algorithmic_bytes_per_launch": launch_bytes}
    cpu = None
    if not a.no_cpu_baseline:
        # the oracle's LM (or ICP) of each agent from the same starts, one agent per host thread,
        # on the first frame (a bounded sample: every agent once)
        import oracle
        from concurrent.futures import ThreadPoolExecutor
        oracle.build()
        om = oracle.OracleMap(mesh.vertices, mesh.faces, mesh.labels)
        sc0 = scans_for(0)
        host = [(sc0[i].depth.cpu().numpy(), sc0[i].cls.cpu().numpy()) for i in range(n_agents)]
        start0 = np.stack([synth.perturb_fixed(truth[0, i], np.random.Generator(np.random.PCG64(a.seed + 11 + i)),
                                               0.10, 1.0) for i in range(n_agents)])

        def orc(i):
            cam = cams[kinds[i]]
            if a.method == "icp":
                return om.icp_align(start0[i], cam, *host[i], 0.3, max_iters=5, step_tol=1e-4)
            return om.align(start0[i], cam, *host[i], max_iters=5)

        cores = os.cpu_count() or 1
        with ThreadPoolExecutor(max_workers=cores) as pool:
            t0 = time.perf_counter()
            list(pool.map(orc, range(n_agents)))
            dt = time.perf_counter() - t0
        cpu = {"value": n_agents / dt, "unit": "scan frames/s", "cores": cores, "kind": "oracle",
               "sample": f"one frame of {n_agents} agents (each 5 iterations), one agent per host thread, "
                         f"{dt:.1f} s wall"}
    print(json.dumps({
        "metric": ("tracking frames/s (64 mixed scans, 5 LM iterations each, 2M-triangle map)" if a.method == "lm"
                   else "tracking frames/s (64 mixed scans, 5 point-to-plane ICP iterations each, 2M-triangle map)"),
        "value": value, "unit": "scan frames/s", "n_gpus": 1, "steps": a.frames, "warmup": 1,
        "ms_per_step": total_ms / a.frames, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": w["name"], "method": a.method, "agents": n_agents, "frames": a.frames,
                   "triangles": mesh.n_tris, "sensors": ["160x120", "640x480", "1024x64 lidar"],
                   "pose_evals": evals, "pose_evals_per_s": evals / (total_ms * 1e-3),
                   "plain_per_pose_frames_per_s": plain_value, "batched_over_plain": value / plain_value,
                   "median_pos_err_m_all_frames": float(np.median(errs)),
                   "agents_within_0.1m_last_frame": float(np.mean(errs[-1] < 0.1)),
                   "agents_within_0.1m_all_frames": float(np.mean(np.all(errs < 0.1, axis=0)))},
        "roofline": roofline, "cpu_baseline": cpu,
        "gpu_launches": a.frames}))


def oracle_row_timings(w, dstart, tol=0.1):
    """The oracle, as it stands, on one unit of each widened row of the 1M-triangle room
    (single thread; a bounded sample each): ICP terms of one pose, the derivative-free search
    from dstart, one meshification, the Eq. 2 normals of one image, the vertex gradient of one
    pose. Seconds per unit."""
    import oracle
    oracle.build()
    mesh, cam = w["mesh"], w["cam"]
    sd, sc = w["scan"]
    om = oracle.OracleMap(mesh.vertices, mesh.faces, mesh.labels)
    out = {}

    def clock(fn):
        t0 = time.perf_counter()
        r = fn()
        return time.perf_counter() - t0, r

    out["icp_terms_s_per_pose"], _ = clock(lambda: om.icp_terms(w["poses"][0], cam, sd, sc, tol))
    dt, (_, rep) = clock(lambda: om.dfo_align(dstart, cam, sd, sc, dfo=oracle.dfo_params(nm_iters=60, cd_iters=40)))
    out["dfo_align_s"] = dt
    out["dfo_evals"] = rep["evals"]
    out["dfo_e_table_final"] = rep["e_table"]
    out["meshify_s_per_image"], _ = clock(lambda: oracle.meshify(cam, sd, sc, w["gt"], cam.range_max, 0.1, 1))
    out["normals_s_per_image"], _ = clock(lambda: oracle.depth_normals(sd, sc, sigma=1.5, metric=True,
                                                                        fx=cam.fx, fy=cam.fy))
    out["vertex_grad_s_per_pose"], _ = clock(lambda: om.vertex_grad(w["poses"][0], cam, sd, sc))
    out["cores"] = 1
    return out


def run_icp(a):
    """Render-accelerated point-to-plane ICP (Sec. V). Value: ICP term evaluations per second
    (render + projective association + J^T e, J^T J) for the 256 candidate poses of the
    1M-triangle 640x480 room, L2 flushed between steps. Alongside: rm_icp_align wall time on
    that room's scan from a 5 cm / 2 deg start and on the 2M-triangle 1024x64 lidar scan
    from its 30 cm / 3 deg start, and the oracle's ICP terms on the host."""
    import ctypes

    import torch
    import paper_1702_06813_gb300 as rm
    from paper_1702_06813_gb300 import _native as N
    import synth
    import __graft_entry__
    __graft_entry__.build_library()
    torch.cuda.set_device(0)
    tol = 0.1
    w = synth.workload_headline(a.seed, a.poses)
    mesh, cam = w["mesh"], w["cam"]
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    intr = rm.Intrinsics.from_camera(cam)
    scan = rm.Scan.make(intr, *w["scan"])
    poses = torch.as_tensor(w["poses"].reshape(-1, 16), dtype=torch.float64, device="cuda")
    n = poses.shape[0]
    gm.set_tuning(tile=(64, 32), wave_poses=min(n, 128))
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")

    def step():
        return rm.icp_terms(gm, scan, poses, tol=tol)

    for _ in range(max(3, a.warmup)):
        out = step()
    torch.cuda.synchronize()

    def timed(fn, k_steps, profile=False):
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(k_steps)]
        torch.cuda.synchronize()
        if profile:
            gm.profile(True)
        for k in range(k_steps):
            flush.fill_(k & 0xFF)
            evs[k][0].record(stream)
            fn()
            evs[k][1].record(stream)
        torch.cuda.synchronize()
        prof = None
        if profile:
            prof = gm.profile_read()
            gm.profile(False)
        return sum(e0.elapsed_time(e1) for e0, e1 in evs), prof

    uuid = None
    try:
        uuid = str(torch.cuda.get_device_properties(0).uuid)
        uuid = uuid if uuid.startswith("GPU-") else "GPU-" + uuid
    except Exception:
        pass
    for attempt in range(2):
        clk = Clocks(uuid)
        clk.start()
        ms, _ = timed(step, a.steps)
        clocks = clk.stop()
        if not {"hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown"} & set(clocks["reasons"]):
            break
    clocks["remeasured"] = attempt > 0
    value = n * a.steps / (ms * 1e-3)
    _, prof = timed(step, a.steps, profile=True)

    # end to end through the C ABI with pinned host poses, scan and outputs
    hp = torch.as_tensor(w["poses"].reshape(-1, 16)).pin_memory()
    hd = torch.as_tensor(w["scan"][0]).pin_memory()
    hc = torch.as_tensor(w["scan"][1]).pin_memory()
    o_n = torch.empty(n, dtype=torch.int64).pin_memory()
    o_l1 = torch.empty(n, dtype=torch.float64).pin_memory()
    o_e2 = torch.empty(n, dtype=torch.float64).pin_memory()
    o_g = torch.empty((n, 6), dtype=torch.float64).pin_memory()
    o_h = torch.empty((n, 21), dtype=torch.float64).pin_memory()
    cs = N.rm_scan(intr.c(), hd.data_ptr(), hc.data_ptr())
    cout = N.rm_icp_out(o_n.data_ptr(), o_l1.data_ptr(), o_e2.data_ptr(), o_g.data_ptr(), o_h.data_ptr())
    sp = ctypes.c_void_p(stream.cuda_stream)

    def e2e_step():
        N.check(N.lib().rm_icp_terms(gm.handle, ctypes.byref(cs), ctypes.c_void_p(hp.data_ptr()), n,
                                     tol, ctypes.byref(cout), sp))

    for _ in range(2):
        e2e_step()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(a.steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_value = n * a.steps / (time.perf_counter() - t0)
    ok = bool(torch.equal(o_n, out["n_assoc"].cpu()) and torch.equal(o_e2, out["e2"].cpu()))

    # alignments: wall time of one rm_icp_align call (host report read back included)
    def align_stats(m, sc, start, gt, tol_a, step_tol, reps=5):
        m_pose, rep = rm.icp_align(m, sc, start, tol=tol_a, max_iters=30, step_tol=step_tol)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(reps):
            m_pose, rep = rm.icp_align(m, sc, start, tol=tol_a, max_iters=30, step_tol=step_tol)
        dt = (time.perf_counter() - t0) / reps
        err = float(np.linalg.norm(m_pose[:3, 3] - gt[:3, 3]))
        return {"ms_per_alignment": dt * 1e3, "iters": rep["iters"], "converged": rep["converged"],
                "n_assoc": rep["n_assoc"], "pos_err_m": err, "tol_m": tol_a, "step_tol": step_tol}

    # the room seen tilted 25 deg toward the floor (a level view of this room leaves one
    # direction unconstrained for point-to-plane ICP: J^T J is singular there)
    rng = np.random.Generator(np.random.PCG64(a.seed + 5))
    gt_room = synth.pose_from(w["gt"][:3, 3], 0.7, math.radians(25.0), 0.0)
    sc_room = rm.Scan.make(intr, *synth.synth_scan(mesh, cam, gt_room, rng, sigma_rel=0.005))
    room_align = align_stats(gm, sc_room, synth.perturb_fixed(gt_room, rng, 0.05, 2.0), gt_room, 0.2, 1e-5)
    # lidar ranges reach 80 m, where FP32 depth steps are ~4e-6 m: the step test sits at 1e-4
    wl = synth.workload_lidar()
    gl = rm.Map(wl["mesh"].vertices, wl["mesh"].faces, wl["mesh"].labels)
    sl = rm.Scan.make(rm.Intrinsics.from_camera(wl["cam"]), *wl["scan"])
    lidar_align = align_stats(gl, sl, wl["start"], wl["gt"], 0.5, 1e-4)
    gl.set_tuning(tile=(16, 16))  # one pose: 4x the tiles of the default 32x32 spread it wider
    lidar_align["tile16x16"] = align_stats(gl, sl, wl["start"], wl["gt"], 0.5, 1e-4)
    gl.close()

    # Eq. 2 normals of 64 depth images (the room scan with per-image noise), sigma 1.5 px,
    # metric: HBM-bound, 17 algorithmic bytes per pixel (depth, class, normal)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(a.seed)
    d0 = torch.as_tensor(w["scan"][0], device="cuda")
    dimg = (d0[None] * (1 + 0.005 * torch.randn((64,) + d0.shape, device="cuda", generator=gen))).contiguous()
    cimg = torch.as_tensor(w["scan"][1], device="cuda")[None].expand(64, -1, -1).contiguous()
    nrm = torch.empty(dimg.shape + (3,), dtype=torch.float32, device="cuda")
    ci = intr.c()

    def normals_step():
        N.check(N.lib().rm_depth_normals(ctypes.byref(ci), 64, ctypes.c_void_p(dimg.data_ptr()),
                                         ctypes.c_void_p(cimg.data_ptr()), 1.5, 1,
                                         ctypes.c_void_p(nrm.data_ptr()), None, sp))

    for _ in range(3):
        normals_step()
    ms_n, _ = timed(normals_step, 20)
    pk, pk_kind = peaks()
    nb = 17 * dimg.numel()
    normals_gbs = nb * 20 / (ms_n * 1e-3) / 1e9
    normals_line = {"images": 64, "image": [cam.width, cam.height], "sigma_px": 1.5, "metric": True,
                    "us_per_launch": ms_n / 20 * 1e3, "images_per_s": 64 * 20 / (ms_n * 1e-3),
                    "algorithmic_bytes_per_launch": nb, "achieved_gbs": normals_gbs,
                    "hbm_frac": normals_gbs / pk["hbm_gbs"],
                    "l2": "flushed between launches (256 MiB write)"}

    # meshification of the room scan (Sec. IV.A): 640x480 -> 306k vertices, 612k faces
    P_img = cam.width * cam.height
    mv = torch.empty((P_img, 3), dtype=torch.float32, device="cuda")
    mf = torch.empty((2 * (cam.width - 1) * (cam.height - 1), 3), dtype=torch.int32, device="cuda")
    ml = torch.empty(mf.shape[0], dtype=torch.uint8, device="cuda")
    mn = torch.empty(1, dtype=torch.int64, device="cuda")
    dscan = rm.Scan.make(intr, *w["scan"])
    dcs = dscan.c()
    gt_dev = torch.as_tensor(w["gt"].reshape(16), dtype=torch.float64, device="cuda")
    mprm = N.rm_meshify_params(cam.range_max, 0.1, 1, 0)

    def mesh_step():
        N.check(N.lib().rm_meshify(ctypes.byref(dcs), ctypes.c_void_p(gt_dev.data_ptr()), ctypes.byref(mprm),
                                   ctypes.c_void_p(mv.data_ptr()), ctypes.c_void_p(mf.data_ptr()),
                                   ctypes.c_void_p(ml.data_ptr()), ctypes.c_void_p(mn.data_ptr()), sp))

    for _ in range(3):
        mesh_step()
    ms_m, _ = timed(mesh_step, 20)
    nfaces = int(mn.item())
    mbytes = 5 * P_img + 12 * P_img + 13 * nfaces
    mesh_line = {"image": [cam.width, cam.height], "faces": nfaces, "us_per_call": ms_m / 20 * 1e3,
                 "algorithmic_bytes": mbytes, "achieved_gbs": mbytes * 20 / (ms_m * 1e-3) / 1e9,
                 "kernels_per_call": 2}

    # derivative-free alignment on the Table I cost (Sec. IV.C), room scan from 3 cm / 1.5 deg
    rng2 = np.random.Generator(np.random.PCG64(a.seed + 9))
    dstart = synth.perturb_fixed(w["gt"], rng2, 0.03, 1.5)
    dpar = rm.dfo_params(nm_iters=60, cd_iters=40)
    rm.dfo_align(gm, scan, dstart, dfo=dpar)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    reps_d = 3
    for _ in range(reps_d):
        dpose, drep = rm.dfo_align(gm, scan, dstart, dfo=dpar)
    dfo_ms = (time.perf_counter() - t0) / reps_d * 1e3
    dfo_line = {"ms_per_alignment": dfo_ms, "evals": drep["evals"], "us_per_eval": dfo_ms * 1e3 / drep["evals"],
                "nm_iters": drep["nm_iters"], "cd_iters": drep["cd_iters"], "converged": drep["converged"],
                "e_table_initial": drep["e_table_initial"], "e_table_final": drep["e_table_final"],
                "pos_err_m": float(np.linalg.norm(dpose[:3, 3] - w["gt"][:3, 3])),
                "batch_slots": 12}
    # the same search with Powell's method in place of Nelder-Mead
    ppar = rm.dfo_params(method="powell", powell_iters=20, cd_iters=40)
    rm.dfo_align(gm, scan, dstart, dfo=ppar)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(reps_d):
        ppose, prep = rm.dfo_align(gm, scan, dstart, dfo=ppar)
    pw_ms = (time.perf_counter() - t0) / reps_d * 1e3
    dfo_line["powell"] = {"ms_per_alignment": pw_ms, "evals": prep["evals"],
                          "us_per_eval": pw_ms * 1e3 / prep["evals"], "powell_iters": prep["powell_iters"],
                          "cd_iters": prep["cd_iters"], "converged": prep["converged"],
                          "e_table_final": prep["e_table_final"],
                          "pos_err_m": float(np.linalg.norm(ppose[:3, 3] - w["gt"][:3, 3]))}

    # Fig. 7's cost landscape: 101-sample sweeps along each of the six twist axes
    def sweeps():
        return [rm.cost_sweep(gm, scan, w["gt"], ax, 0.3 if ax < 3 else 0.1, 101) for ax in range(6)]

    sweeps()
    ms_s, _ = timed(sweeps, 3)
    sweep_line = {"axes": 6, "samples_per_axis": 101, "span": [0.3, 0.3, 0.3, 0.1, 0.1, 0.1],
                  "ms_per_six_sweeps": ms_s / 3, "pose_evals_per_s": 606 * 3 / (ms_s * 1e-3)}

    # vertex-position gradient summed over 16 candidate poses (map refinement)
    vposes = poses[:16]
    rm.cost_grad_vertices(gm, scan, vposes)
    ms_v, _ = timed(lambda: rm.cost_grad_vertices(gm, scan, vposes), 5)
    vgrad_line = {"poses": 16, "vertices": mesh.n_verts, "ms_per_call": ms_v / 5,
                  "pose_evals_per_s": 16 * 5 / (ms_v * 1e-3),
                  "note": "render with ids and barycentrics, then FP64 atomics per active pixel"}

    P = cam.width * cam.height
    ab = algorithmic_bytes(mesh.n_verts, mesh.n_tris, P)
    kern = prof["kernels"]
    dom = max(kern, key=lambda k: kern[k][1])
    launches, tot = kern[dom]
    per_launch = n * a.steps / launches
    avg_s = tot * 1e-3 / launches
    achieved = ab[dom] * per_launch / avg_s / 1e9
    share = {k: round(v[1] / sum(x[1] for x in kern.values()), 4) for k, v in kern.items()}
    line = {
        "metric": "ICP term evals/s (render + projective association + point-to-plane J^T e, J^T J) "
                  "640x480, 1M tris",
        "value": value, "unit": "pose evals/s", "n_gpus": 1, "steps": a.steps,
        "warmup": max(3, a.warmup), "ms_per_step": ms / a.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": w["name"] + "-icp", "poses_per_gpu": n, "triangles": mesh.n_tris,
                   "image": [cam.width, cam.height], "tol_m": tol, "tile": [64, 32],
                   "wave_poses": min(n, 128), "l2": "flushed between timed steps (256 MiB write)",
                   "kernel_share": share, "e2e_matches_device": ok,
                   "align_room_1M_640x480": room_align, "align_lidar_2M_1024x64": lidar_align,
                   "depth_normals_eq2": normals_line, "meshify_sec4a": mesh_line,
                   "dfo_align_table1_room": dfo_line, "vertex_grad": vgrad_line, "cost_sweep_fig7": sweep_line,
                   "step_hbm_roofline_frac": step_algorithmic_bytes(mesh.n_verts, mesh.n_tris, P, n, min(n, 128))
                   * a.steps / (ms * 1e-3) / 1e9 / pk["hbm_gbs"]},
        "clocks": clocks,
        "e2e": {"value": e2e_value, "unit": "pose evals/s",
                "h2d_bytes_per_step": int(hp.numel() * 8 + hd.numel() * 4 + hc.numel()),
                "d2h_bytes_per_step": int(n * (8 + 8 + 8 + 48 + 168))},
        "gpu_launches": int(prof["launches"] // a.steps) * a.steps,
        "roofline": {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": pk["hbm_gbs"],
                     "unit": "GB/s", "frac": achieved / pk["hbm_gbs"], "traffic": None,
                     "peak_kind": pk_kind, "avg_launch_ms": avg_s * 1e3, "poses_per_launch": per_launch},
    }
    if not a.no_cpu_baseline:
        import oracle
        oracle.build()
        om = oracle.OracleMap(mesh.vertices, mesh.faces, mesh.labels)
        sd, sc = w["scan"]
        om.icp_terms(w["poses"][0], cam, sd, sc, tol)
        from concurrent.futures import ThreadPoolExecutor
        cores = os.cpu_count() or 1
        with ThreadPoolExecutor(max_workers=cores) as pool:  # the oracle's C calls drop the GIL
            done = 0
            t0 = time.perf_counter()
            while time.perf_counter() - t0 < 2.0:
                list(pool.map(lambda k: om.icp_terms(w["poses"][k], cam, sd, sc, tol), range(n)))
                done += n
            dt = time.perf_counter() - t0
        line["cpu_baseline"] = {"value": done / dt, "unit": "pose evals/s", "cores": cores, "kind": "oracle",
                                "sample": f"{done // n} pass(es) over the {n} candidate poses, one pose per "
                                          f"host thread, {dt:.1f} s wall"}
        line["config"]["oracle_per_row"] = oracle_row_timings(w, dstart, tol)
    print(json.dumps(line))
    gm.close()


def _timed_events(fn, steps, flush):
    """Total milliseconds of `steps` calls of fn on the current stream, the L2 flushed (a
    256 MiB write) before each, CUDA events around each call."""
    import torch
    stream = torch.cuda.current_stream()
    tot = 0.0
    for k in range(steps):
        flush.fill_(k & 0xFF)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fn()
        e1.record(stream)
        torch.cuda.synchronize()
        tot += e0.elapsed_time(e1)
    return tot


def _small_line(a, metric, unit, value, ms, config, roofline, cpu, launches):
    print(json.dumps({
        "metric": metric, "value": value, "unit": unit, "n_gpus": 1, "steps": a.steps,
        "warmup": max(3, a.warmup), "ms_per_step": ms / a.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": config,
        "roofline": roofline, "cpu_baseline": cpu, "gpu_launches": launches}))


def run_lidar(a):
    """The panoramic workload: cost and gradient of 64 candidate poses (30 cm / 3 deg around the
    true pose) through the 1024 x 64 ray table on the 2M-triangle terrain (render + Table I +
    surrogate + adjoint), one rm_cost_grad call per step with the default tiles; then LM
    alignment from the 30 cm / 3 deg start. The raster's algorithmic bytes are the scan's, 5 per ray per pose. CPU
    baseline: the oracle over 16 of the poses on the host cores."""
    import torch
    import paper_1702_06813_gb300 as rm
    import synth
    import __graft_entry__
    __graft_entry__.build_library()
    torch.cuda.set_device(0)
    w = synth.workload_lidar(a.seed + 4000)
    mesh, cam = w["mesh"], w["cam"]
    n = 64
    r = np.random.Generator(np.random.PCG64(a.seed + 41))
    poses_np = synth.perturb_gauss(w["gt"], r, 0.3, 3.0, n)
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    scan = rm.Scan.make(rm.Intrinsics.from_camera(cam), *w["scan"])
    poses = torch.as_tensor(poses_np.reshape(-1, 16), dtype=torch.float64, device="cuda")
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    if a.tile:  # default: the ray-table tile (16x16); large tiles grow panoramic bins a lot
        tw, th = (int(x) for x in a.tile.split("x"))
        gm.set_tuning(tile=(tw, th))
    for _ in range(max(3, a.warmup)):
        rm.cost_grad(gm, scan, poses)
    torch.cuda.synchronize()
    ms = _timed_events(lambda: rm.cost_grad(gm, scan, poses), a.steps, flush)
    gm.profile(True)
    _timed_events(lambda: rm.cost_grad(gm, scan, poses), a.steps, flush)
    prof = gm.profile_read()
    gm.profile(False)
    tune = gm.get_tuning()
    kms = {k: v[1] / a.steps for k, v in prof["kernels"].items()}
    P = cam.width * cam.height
    wave = tune["wave_poses"] if tune["wave_poses"] > 0 else n
    waves = -(-n // wave)
    rl_ms = kms.get("k_raster", 0.0) / waves
    pk, pk_kind = peaks()
    achieved = 5 * P * min(n, wave) / (rl_ms * 1e-3) / 1e9 if rl_ms > 0 else None
    # LM alignment from the 30 cm / 3 deg start (the configuration's own task)
    rm.align(gm, scan, w["start"], max_iters=50)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    pose, rep_lm = rm.align(gm, scan, w["start"], max_iters=50)
    lm_ms = (time.perf_counter() - t0) * 1e3
    cpu = None
    if not a.no_cpu_baseline:
        import oracle
        oracle.build()
        om = oracle.OracleMap(mesh.vertices, mesh.faces, mesh.labels)
        t0 = time.perf_counter()
        res = om.cost_batch(poses_np[:16], cam, *w["scan"])
        dt = time.perf_counter() - t0
        cpu = {"value": 16 / dt, "unit": "pose evals/s", "cores": int(res["threads"]), "kind": "oracle",
               "sample": f"16 of the 64 poses, OpenMP over poses, {dt:.1f} s wall"}
    _small_line(a, "Lidar pose evals/s (render+residual+grad) 1024x64 ray table, 2M tris", "pose evals/s",
                n * a.steps / (ms * 1e-3), ms,
                {"workload": w["name"] + "-64poses", "poses_per_step": n, "triangles": mesh.n_tris,
                 "rays": [cam.width, cam.height], "tile": list(tune["tile"]), "wave_poses": tune["wave_poses"],
                 "kernel_ms_per_step": kms, "l2": "flushed between timed steps (256 MiB write)",
                 "lm_align_from_30cm_3deg": {"ms": lm_ms, "iters": rep_lm["iters"],
                                             "converged": rep_lm["converged"],
                                             "pos_err_m": float(np.linalg.norm(pose[:3, 3] - w["gt"][:3, 3]))}},
                {"bound": "hbm", "kernel": "k_raster", "achieved": achieved, "peak": pk["hbm_gbs"],
                 "unit": "GB/s", "frac": (achieved / pk["hbm_gbs"]) if achieved else None, "traffic": None,
                 "peak_kind": pk_kind, "avg_launch_ms": rl_ms, "poses_per_launch": min(n, wave)},
                cpu, int(prof["launches"]))
    gm.close()


def run_normals(a):
    """Eq. 2 surface normals (Sec. V) of 64 noisy copies of the 640x480 room scan per step
    (sigma 1.5 px, metric), one rm_depth_normals call. Algorithmic bytes: depth and class in,
    the normal out, 17 per pixel. CPU baseline: the oracle on one image per host thread."""
    import torch
    import paper_1702_06813_gb300 as rm
    import synth
    import __graft_entry__
    __graft_entry__.build_library()
    torch.cuda.set_device(0)
    w = synth.workload_headline(a.seed, 1)
    cam = w["cam"]
    intr = rm.Intrinsics.from_camera(cam)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(a.seed)
    d0 = torch.as_tensor(w["scan"][0], device="cuda")
    D = (d0[None] * (1 + 0.005 * torch.randn((64,) + d0.shape, device="cuda", generator=gen))).contiguous()
    C = torch.as_tensor(w["scan"][1], device="cuda")[None].expand(64, -1, -1).contiguous()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(max(3, a.warmup)):
        rm.depth_normals(intr, D, C, sigma=1.5, metric=True)
    torch.cuda.synchronize()
    ms = _timed_events(lambda: rm.depth_normals(intr, D, C, sigma=1.5, metric=True), a.steps, flush)
    pk, pk_kind = peaks()
    nb = 17 * D.numel()
    achieved = nb * a.steps / (ms * 1e-3) / 1e9
    cpu = None
    if not a.no_cpu_baseline:
        import oracle
        from concurrent.futures import ThreadPoolExecutor
        oracle.build()
        Dh, Ch = D[:16].cpu().numpy(), C[:16].cpu().numpy()
        cores = os.cpu_count() or 1
        with ThreadPoolExecutor(max_workers=cores) as pool:
            t0 = time.perf_counter()
            list(pool.map(lambda k: oracle.depth_normals(Dh[k], Ch[k], sigma=1.5, metric=True, fx=cam.fx,
                                                         fy=cam.fy), range(16)))
            dt = time.perf_counter() - t0
        cpu = {"value": 16 / dt, "unit": "images/s", "cores": cores, "kind": "oracle",
               "sample": f"16 of the 64 images, one per host thread, {dt:.1f} s wall"}
    _small_line(a, "Eq. 2 depth-image normals/s (640x480, sigma 1.5 px, metric)", "images/s",
                64 * a.steps / (ms * 1e-3), ms,
                {"workload": "room-scan-640x480-x64-normals", "images_per_step": 64, "sigma_px": 1.5,
                 "l2": "flushed between timed steps (256 MiB write)"},
                {"bound": "hbm", "kernel": "k_depth_normals", "achieved": achieved, "peak": pk["hbm_gbs"],
                 "unit": "GB/s", "frac": achieved / pk["hbm_gbs"], "traffic": None, "peak_kind": pk_kind,
                 "avg_launch_ms": ms / a.steps, "algorithmic_bytes_per_launch": nb},
                cpu, a.steps)


def run_vgrad(a):
    """Vertex-position gradient (map refinement) of 16 candidate poses of the 1M-triangle room
    per step, one rm_cost_grad_vertices call: visibility-buffer render, then the per-pixel
    scatter kernel. Algorithmic bytes per pose: the map (12 V + 13 T, once per call), the scan
    (5 P) and the FP64 gradient (24 V, once per call). CPU baseline: the oracle, one pose per
    host thread."""
    import torch
    import paper_1702_06813_gb300 as rm
    import synth
    import __graft_entry__
    __graft_entry__.build_library()
    torch.cuda.set_device(0)
    w = synth.workload_headline(a.seed, 16)
    mesh, cam = w["mesh"], w["cam"]
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    scan = rm.Scan.make(rm.Intrinsics.from_camera(cam), *w["scan"])
    poses = torch.as_tensor(w["poses"].reshape(-1, 16), dtype=torch.float64, device="cuda")
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(max(3, a.warmup)):
        rm.cost_grad_vertices(gm, scan, poses)
    torch.cuda.synchronize()
    gm.profile(True)
    ms = _timed_events(lambda: rm.cost_grad_vertices(gm, scan, poses), a.steps, flush)
    prof = gm.profile_read()
    gm.profile(False)
    pk, pk_kind = peaks()
    P = cam.width * cam.height
    nb = 12 * mesh.n_verts + 13 * mesh.n_tris + 24 * mesh.n_verts + 16 * 5 * P
    achieved = nb * a.steps / (ms * 1e-3) / 1e9
    cpu = None
    if not a.no_cpu_baseline:
        import oracle
        from concurrent.futures import ThreadPoolExecutor
        oracle.build()
        om = oracle.OracleMap(mesh.vertices, mesh.faces, mesh.labels)
        cores = os.cpu_count() or 1
        with ThreadPoolExecutor(max_workers=cores) as pool:
            t0 = time.perf_counter()
            list(pool.map(lambda k: om.vertex_grad(w["poses"][k], cam, *w["scan"]), range(16)))
            dt = time.perf_counter() - t0
        cpu = {"value": 16 / dt, "unit": "pose evals/s", "cores": cores, "kind": "oracle",
               "sample": f"the 16 poses, one per host thread, {dt:.1f} s wall"}
    _small_line(a, "vertex-gradient pose evals/s (640x480, 1M tris, d e_ls / d vertices)", "pose evals/s",
                16 * a.steps / (ms * 1e-3), ms,
                {"workload": w["name"] + "-vgrad16", "poses_per_step": 16, "vertices": mesh.n_verts,
                 "kernel_ms_per_step": {k: v[1] / a.steps for k, v in prof["kernels"].items()},
                 "l2": "flushed between timed steps (256 MiB write)"},
                {"bound": "hbm", "kernel": "whole call", "achieved": achieved, "peak": pk["hbm_gbs"],
                 "unit": "GB/s", "frac": achieved / pk["hbm_gbs"], "traffic": None, "peak_kind": pk_kind,
                 "avg_launch_ms": ms / a.steps, "algorithmic_bytes_per_call": nb},
                cpu, int(prof["launches"]))
    gm.close()


def main():
    a = args_()
    if a.impl == "reference":
        run_reference(a)
        return
    if a.workload == "tracking":
        run_tracking(a)
        return
    if a.workload == "icp":
        run_icp(a)
        return
    if a.workload == "normals":
        run_normals(a)
        return
    if a.workload == "vgrad":
        run_vgrad(a)
        return
    if a.workload == "lidar":
        run_lidar(a)
        return
    import torch
    import torch.distributed as dist

    world, rank, local = rank_info()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    def barrier():
        if world > 1:
            dist.barrier()

    import __graft_entry__
    __graft_entry__.build_library()
    import ctypes

    import paper_1702_06813_gb300 as rm
    from paper_1702_06813_gb300 import _native as N
    import synth

    w = synth.workload_headline(rank_seed(a.seed, rank), a.poses)
    mesh, cam = w["mesh"], w["cam"]
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    intr = rm.Intrinsics.from_camera(cam)
    scan = rm.Scan.make(intr, *w["scan"])
    poses = torch.as_tensor(w["poses"].reshape(-1, 16), dtype=torch.float64, device="cuda")
    n = poses.shape[0]
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")  # > 129 MB L2

    def step():
        return rm.cost_grad(gm, scan, poses)

    from paper_1702_06813_gb300 import autotune
    if a.tile:
        tw, th = (int(x) for x in a.tile.split("x"))
        gm.set_tuning(tile=(tw, th), wave_poses=min(n, 128))
        tuned = {"ms": None}
    else:
        tuned = autotune.autotune(gm, scan, poses, cache=None, reps=3)  # untimed: part of warm-up
    for _ in range(max(3, a.warmup)):
        out = step()
    torch.cuda.synchronize()
    tune = gm.get_tuning()

    def timed(fn, k_steps, profile=False):
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(k_steps)]
        barrier()
        torch.cuda.synchronize()
        if profile:
            gm.profile(True)
        for k in range(k_steps):
            flush.fill_(k & 0xFF)
            evs[k][0].record(stream)
            fn()
            evs[k][1].record(stream)
        torch.cuda.synchronize()
        barrier()
        ms = sum(e0.elapsed_time(e1) for e0, e1 in evs)
        prof = None
        if profile:
            prof = gm.profile_read()
            gm.profile(False)
        return ms, prof

    uuid = None
    try:
        uuid = str(torch.cuda.get_device_properties(local).uuid)
        uuid = uuid if uuid.startswith("GPU-") else "GPU-" + uuid
    except Exception:
        pass
    for attempt in range(2):
        clk = Clocks(uuid)
        clk.start()
        ms, _ = timed(step, a.steps)
        clocks = clk.stop()
        bad = {"hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown"} & set(clocks["reasons"])
        if not bad:
            break
    clocks["remeasured"] = attempt > 0
    ms = max_over_ranks(ms, world, "cuda")
    ms_per_step = ms / a.steps
    value = job_rate(world, n * a.steps, ms * 1e-3)
    # per-kernel durations: the same steps again with the library's event profiler on (its
    # waves then run on one stream, so each kernel's interval is its own)
    _, prof = timed(step, a.steps, profile=True)

    # plain form: one pose per call
    def plain():
        for i in range(n):
            rm.cost_grad(gm, scan, poses[i:i + 1])
    plain_steps = max(1, min(3, a.steps))
    ms_plain, _ = timed(plain, plain_steps)
    plain_value = n * plain_steps / (ms_plain * 1e-3)

    # the batch entry point on the same poses
    rm.cost_grad_batch(gm, scans=scan, poses=poses)
    ms_batch, _ = timed(lambda: rm.cost_grad_batch(gm, scans=scan, poses=poses), a.steps)
    batch_value = n * a.steps / (ms_batch * 1e-3)

    # end to end through the C ABI with pinned host buffers
    hp = torch.empty((n, 16), dtype=torch.float64).pin_memory()
    hp.copy_(torch.as_tensor(w["poses"].reshape(-1, 16)))
    hd = torch.as_tensor(w["scan"][0]).pin_memory()
    hc = torch.as_tensor(w["scan"][1]).pin_memory()
    o_counts = torch.empty((n, 6), dtype=torch.int64).pin_memory()
    o_et = torch.empty(n, dtype=torch.int64).pin_memory()
    o_els = torch.empty(n, dtype=torch.float64).pin_memory()
    o_g = torch.empty((n, 6), dtype=torch.float64).pin_memory()
    o_h = torch.empty((n, 21), dtype=torch.float64).pin_memory()
    cs = N.rm_scan(intr.c(), hd.data_ptr(), hc.data_ptr())
    cout = N.rm_cost_out(o_counts.data_ptr(), o_et.data_ptr(), o_els.data_ptr(), o_g.data_ptr(), o_h.data_ptr())
    prm = rm.cost_params()
    sp = ctypes.c_void_p(stream.cuda_stream)

    def e2e_step():
        N.check(N.lib().rm_cost_grad(gm.handle, ctypes.byref(cs), ctypes.c_void_p(hp.data_ptr()), n,
                                     ctypes.byref(prm), ctypes.byref(cout), sp))

    for _ in range(2):
        e2e_step()
    barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(a.steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    e2e_value = job_rate(world, n * a.steps, max_over_ranks(e2e_s, world, "cuda"))
    h2d = hp.numel() * 8 + hd.numel() * 4 + hc.numel()
    d2h = n * (6 * 8 + 8 + 8 + 6 * 8 + 21 * 8)
    # sanity: the e2e numbers equal the device path's
    ok = bool(torch.equal(o_counts, out["counts"].cpu()) and torch.equal(o_els, out["e_ls"].cpu()))

    # roofline of the dominant kernel
    P = cam.width * cam.height
    ab = algorithmic_bytes(mesh.n_verts, mesh.n_tris, P)
    pk, pk_kind = peaks()
    kern = prof["kernels"]
    dom = max(kern, key=lambda k: kern[k][1])
    launches, tot = kern[dom]
    per_launch_poses = n * a.steps / launches
    avg_s = tot * 1e-3 / launches
    achieved = ab[dom] * per_launch_poses / avg_s / 1e9
    share = {k: round(v[1] / sum(x[1] for x in kern.values()), 4) for k, v in kern.items()}
    step_bytes = step_algorithmic_bytes(mesh.n_verts, mesh.n_tris, P, n, tune["wave_poses"])
    step_frac = step_bytes * a.steps / (ms * 1e-3) / 1e9 / pk["hbm_gbs"]
    dram_raster = measured_traffic(dom, per_launch_poses, mesh.n_tris)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": a.steps,
        "warmup": max(3, a.warmup), "ms_per_step": ms_per_step, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": w["name"], "poses_per_gpu": n, "triangles": mesh.n_tris,
                   "vertices": mesh.n_verts, "image": [cam.width, cam.height],
                   "l2": "flushed between timed steps (256 MiB write)",
                   "tile": list(tune["tile"]), "bin_capacity": tune["bin_capacity"],
                   "wave_poses": tune["wave_poses"], "autotuned_ms": tuned["ms"],
                   "plain_one_pose_per_call_evals_per_s": plain_value,
                   "batch_entry_evals_per_s": batch_value,
                   "batched_over_plain": value / plain_value,
                   "algorithmic_mb_per_eval": ab["total"] / 1e6,
                   "step_algorithmic_mb_map_once_per_wave": step_bytes / 1e6,
                   "step_hbm_roofline_frac": step_frac,
                   "raster_dram_mb_per_eval_ncu": (dram_raster / per_launch_poses / 1e6
                                                   if dram_raster else None),
                   "kernel_share": share, "e2e_matches_device": ok},
        "clocks": clocks,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)},
        "gpu_launches": int(prof["launches"] // a.steps) * a.steps,
        "roofline": {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": pk["hbm_gbs"],
                     "unit": "GB/s", "frac": achieved / pk["hbm_gbs"],
                     "traffic": dram_raster,
                     "peak_kind": pk_kind, "avg_launch_ms": avg_s * 1e3,
                     "poses_per_launch": per_launch_poses},
    }
    if rank == 0 and world == 1 and not a.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w)
        line["config"]["oracle_single_thread_evals_per_s"] = oracle_single_thread(w)
    if rank == 0:
        print(json.dumps(line))
    gm.close()
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
