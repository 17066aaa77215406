"""Benchmark: projective TSDF integration of the 640x480 room sequence.

Workload: the seeded 10x10x3 m room, 300 frames of 640x480 float32 depth
(f = 525, noise N(0, (0.0012 z^2)^2), 5 % invalid pixels, depth > 5 m
invalid), voxel 0.02 m, truncation 4 voxels, max weight 100, FP32 storage.
One step = every step of the integration path over the whole sequence into a
freshly reset map: band-segment block allocation in the GPU hash, then the
per-voxel projective TSDF update, frames batched `--batch` per launch.

Prints one JSON line (rank 0).  `value` is voxel updates per second over all
ranks (each rank integrates its own replica: the path shards by map, no
collective); `e2e` repeats the measurement with depth frames copied from
pinned host memory inside the timed region.  `--impl reference` times the
CPU oracle (test infrastructure, FP64) on a bounded sample of the same
workload instead.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "TSDF voxel updates/s and frames/s (640x480, 2 cm); % HBM peak; p99 latency"
UNIT = "voxel updates/s"
WORKLOAD = "room 10x10x3 m, 300 frames 640x480 f=525, voxel 0.02 m, trunc 4 voxels, max weight 100"


# GB300: 152 SMs x 128 FP32/INT32 lanes at the 2070 MHz maximum SM clock
ALU_PEAK_OPS = 152 * 128 * 2.070e9
# algorithmic ALU operations of the allocator's prescribed decision sequence:
# per band segment (ray direction 6, band ends 3, start point 3, range check 3,
# floor and convert 6, three axes x (sign 2, reciprocal 1, boundary 1,
# crossing 2) = 18, key 7) and per emitted cell (axis choice 4, end test 2,
# advance 4, duplicate check 2)
OPS_PER_SEGMENT = 46
OPS_PER_CELL = 12
# algorithmic operations of one voxel projection and update (pinhole, FP32):
# voxel x coordinate 2, position 3, reciprocal depth 1, pixel 6, in-image 5,
# pixel index 3, depth load 1, d_p 1, validity 3, update (clamp, weight sum,
# difference, quotient 2, sum, cap) 7
OPS_PER_PROJECTION = 32


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            pk = json.load(fh)
        return float(pk["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def _kernel_rev() -> str:
    import hashlib
    with open(os.path.join(ROOT, "paper_2311_00626_gb300", "csrc", "kernels.cu"), "rb") as fh:
        return hashlib.sha1(fh.read()).hexdigest()[:12]


def _traffic(kernel: str):
    """DRAM bytes per launch of `kernel` from the committed ncu record, if it
    was taken on the current kernels.cu; else None."""
    path = os.path.join(ROOT, "profiles", "ncu_traffic.txt")
    try:
        rev = _kernel_rev()
        with open(path) as fh:
            for line in fh:
                f = line.split()
                if (len(f) >= 3 and not line.startswith("#") and f[0] == rev
                        and f[1].split("<")[0] == kernel):
                    return float(f[2])
    except OSError:
        pass
    return None


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.dev}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for name, val in zip(names, f[5:9]):
                if val.lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "samples": len(sm),
                "reasons": sorted(reasons)}


def reduce_max(x: float, ws: int, device: str = "cuda") -> float:
    """Max of a per-rank scalar over all ranks (the job's time is its slowest
    rank's); the identity for a single process."""
    if ws <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate_rate(work_per_rank: float, ms_max: float, ws: int) -> float:
    """Whole-job throughput of `ws` replicas each doing `work_per_rank` units,
    timed by the slowest rank."""
    return ws * work_per_rank / (ms_max * 1e-3)


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def reference_arm(args):
    """Time the CPU oracle on a bounded sample of the workload (rank 0)."""
    ws, rank, _ = _dist()
    if rank != 0:
        return
    import oracle
    import synth
    w = synth.config_room(n_frames=300)
    # size the per-step sample so that warm-up plus timed steps take about
    # two minutes of host time
    probe = oracle.OracleMap(w.voxel_size, w.truncation_voxels, w.max_weight)
    t0 = time.perf_counter()
    for f in w.frames[:10]:
        probe.integrate(f.sensor, f.T, f.depth)
    per_frame = (time.perf_counter() - t0) / 10
    probe.close()
    n = int(min(300, max(10, 120.0 / ((args.warmup + args.steps) * per_frame))))
    per_step = []
    updates = 0
    for step in range(args.warmup + args.steps):
        m = oracle.OracleMap(w.voxel_size, w.truncation_voxels, w.max_weight)
        t0 = time.perf_counter()
        for f in w.frames[:n]:
            m.integrate(f.sensor, f.T, f.depth)
        dt = time.perf_counter() - t0
        updates = m.counters()["total_updates"]
        m.close()
        if step >= args.warmup:
            per_step.append(dt)
    sec = sum(per_step)
    value = updates * len(per_step) / sec
    cores = os.cpu_count()
    sample = f"first {n} of 300 frames per step (oracle, FP64, OpenMP over blocks)"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * sec / len(per_step), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "sample_frames": n},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0},
            "frames_per_s": n * len(per_step) / sec}
    print(json.dumps(line), flush=True)


def cpu_baseline(frames_n: int):
    import oracle
    import synth
    w = synth.config_room(n_frames=300)
    m = oracle.OracleMap(w.voxel_size, w.truncation_voxels, w.max_weight)
    t0 = time.perf_counter()
    for f in w.frames[:frames_n]:
        m.integrate(f.sensor, f.T, f.depth)
    dt = time.perf_counter() - t0
    upd = m.counters()["total_updates"]
    m.close()
    return {"value": upd / dt, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle",
            "sample": f"first {frames_n} of the 300 frames, one pass ({dt:.1f} s)"}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--batch", type=int, default=300,
                    help="frames per integrate_batch call (sub-batches of 32 per launch pair; "
                         "more than 32 pipelines allocation with integration)")
    ap.add_argument("--ref-frames", type=int, default=300,
                    help="frames of the room sequence the CPU oracle integrates for cpu_baseline "
                         "(the whole 300-frame step takes ~9 s on 16 Grace cores)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-forms", action="store_true")
    ap.add_argument("--workload", default="room", choices=["room", "rig", "serving", "layers"],
                    help="room: the 640x480 sequence (default); rig: 4 cameras + LiDAR per step, "
                         "FP16, CUDA graph; serving: 16 maps, Poisson arrivals, continuous batching; "
                         "layers: ESDF and marching-cubes mesh of the room map, from scratch and "
                         "incremental")
    ap.add_argument("--rig-steps", type=int, default=200)
    ap.add_argument("--serve-seconds", type=float, default=60.0,
                    help="simulated seconds of Poisson arrivals (the paced run takes as long)")
    ap.add_argument("--serve-pool", type=int, default=32, help="distinct poses per map")
    ap.add_argument("--serve-max-blocks", type=int, default=0,
                    help="pool blocks per serving map (0: the library default); smaller maps keep a "
                         "profiler capture of the serving workload within a few GB of device memory")
    ap.add_argument("--launch-shape", default="",
                    help="room launch shape as TILE_H,CTAS_PER_SM (e.g. 32,0) instead of the autotuner's pick; "
                         "for profiling commands, whose launch counts must not depend on the tuning")
    ap.add_argument("--no-rig", action="store_true", help="leave the rig form out of the default line")
    ap.add_argument("--no-serving", action="store_true",
                    help="leave the serving form out of the default line")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    if args.impl == "reference":
        return reference_arm(args)
    if args.workload == "rig":
        return bench_rig(args)
    if args.workload == "serving":
        return bench_serving(args)
    if args.workload == "layers":
        return bench_layers(args)

    ws, rank, local = _dist()
    import numpy as np
    import torch
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    import paper_2311_00626_gb300 as gt
    import synth
    w = synth.config_room(n_frames=300)
    n_frames = len(w.frames)
    host = torch.from_numpy(np.stack([f.depth for f in w.frames])).pin_memory()
    dev = host.to("cuda", non_blocking=False)
    frames_dev = [dev[i] for i in range(n_frames)]
    in_bytes = host.numel() * 4

    def make_step(m, batch):
        descs = [gt.frame_desc(0, f.sensor, f.T, d) for f, d in zip(w.frames, frames_dev)]

        def step():
            m.reset()
            if batch == 1:
                for f, d in zip(w.frames, frames_dev):
                    m.integrate(f.sensor, f.T, d)
            else:
                for s in range(0, n_frames, batch):
                    gt.integrate_batch([m.handle], descs[s:s + batch])
        return step

    def barrier():
        if ws > 1:
            import torch.distributed as dist
            dist.barrier()

    def timed(step, k):
        barrier()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(k):
            step()
        e1.record()
        torch.cuda.synchronize()
        barrier()
        return reduce_max(e0.elapsed_time(e1) / k, ws)

    # ---- launch shape picked by the autotuner (results do not depend on it)
    from paper_2311_00626_gb300.serving import autotune

    def time_shape(cfg):
        mt = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, storage=gt.STORAGE_FP32, **cfg)
        st_ = make_step(mt, args.batch)
        st_()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(3):
            st_()
        b.record()
        torch.cuda.synchronize()
        mt.close()
        return a.elapsed_time(b) / 3

    if args.launch_shape:
        th, cp = (int(x) for x in args.launch_shape.split(","))
        shape, shape_timings = {"alloc_tile_h": th, "integrate_ctas_per_sm": cp}, []
    else:
        shapes = [{"alloc_tile_h": t, "integrate_ctas_per_sm": c} for t in (16, 32) for c in (0, 3, 4, 5)]
        shape, shape_timings = autotune(f"room{args.batch}", time_shape, shapes, cache=False)

    # ---- headline: FP32 storage, batched launches
    m = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, storage=gt.STORAGE_FP32, **shape)
    step = make_step(m, args.batch)
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    # walk statistics (band segments and cells, for the allocator's roofline)
    # from one extra untimed step: counting them costs about 5 %
    gt.map_walk_stats(m.handle, True)
    step()
    walk = m.stats()
    gt.map_walk_stats(m.handle, False)
    st = m.stats()
    updates_per_step = st["voxel_updates"]
    clocks = ClockSampler(local)
    clocks.start()
    ms = timed(step, args.steps)
    clk = clocks.stop()
    # per-kernel event times from a second, separately timed run (the events
    # recorded around every launch would perturb the headline step)
    gt.map_timing(m.handle, True)
    timed(step, args.steps)
    alloc_ms, integ_ms, calls = gt.map_kernel_times(m.handle)
    gt.map_timing(m.handle, False)
    # the same launches timed alone: 32 frames per call, so each call is one
    # sub-batch whose two kernels run one after the other, not overlapped
    iso_step = make_step(m, 32)
    iso_step()
    gt.map_timing(m.handle, True)
    timed(iso_step, max(3, args.steps // 4))
    iso_alloc, iso_integ, iso_calls = gt.map_kernel_times(m.handle)
    gt.map_timing(m.handle, False)
    st = m.stats()
    assert st["voxel_updates"] == updates_per_step, "non-deterministic update count"
    launches_per_step = st["launches"]
    visits = st["block_visits"]
    fresh = st["blocks"]
    # integration kernel, HBM roofline: every listed block read and written
    # once per launch (fresh blocks only written), plus the depth images
    block_bytes = 512 * 8
    bytes_per_step = (2 * visits - fresh) * block_bytes + in_bytes
    integ_bytes_per_launch = bytes_per_step / launches_per_step
    integ_ms_per_launch = integ_ms / max(calls, 1)
    hbm_peak, peak_src = _peaks()
    achieved = integ_bytes_per_launch / (integ_ms_per_launch * 1e-3) / 1e9
    # allocation kernel: the depth images it cannot do without, and the rate of
    # a kernel that would walk every band segment in the same time (it walks
    # about a sixth of them, so that rate is no fraction of a peak)
    alloc_bytes_per_launch = in_bytes / launches_per_step
    alloc_ms_per_launch = alloc_ms / max(calls, 1)
    alloc_ops_per_launch = (OPS_PER_SEGMENT * walk["segments"] + OPS_PER_CELL * walk["cells"]) / launches_per_step
    alloc_gbs = alloc_bytes_per_launch / (alloc_ms_per_launch * 1e-3) / 1e9
    iso_alloc_ms = iso_alloc / max(iso_calls, 1)
    alloc_share = alloc_ms / max(alloc_ms + integ_ms, 1e-9)
    # integration kernel, ALU roofline: 512 voxel projections per (block,
    # frame) pair it integrates
    integ_ops_per_launch = OPS_PER_PROJECTION * 512.0 * st["block_frame_pairs"] / launches_per_step
    integ_alu_achieved = integ_ops_per_launch / (integ_ms_per_launch * 1e-3)
    value = aggregate_rate(updates_per_step, ms, ws)
    fps = aggregate_rate(n_frames, ms, ws)

    # ---- end to end through the public API with host buffers
    # the public call for host images: integrate_batch_host copies each
    # sub-batch's frames from pinned host memory into a staging buffer while
    # the previous sub-batch integrates
    host_descs = [gt.frame_desc_host(0, f.sensor, f.T, host[i]) for i, f in enumerate(w.frames)]
    staging = torch.empty(4 * 32 * host[0].numel() * 4, dtype=torch.uint8, device="cuda")  # 4 slots
    host_res = torch.zeros(6, dtype=torch.int64)

    def e2e_step():
        m.reset()
        for s0 in range(0, n_frames, args.batch):
            gt.integrate_batch_host([m.handle], host_descs[s0:s0 + args.batch], staging)
        s = m.stats()  # device -> host read of the step's result (synchronises)
        host_res[1] = s["voxel_updates"]
        assert s["voxel_updates"] == updates_per_step

    k_e2e = max(1, min(args.steps, 10))
    for _ in range(args.warmup):  # the first call creates the copy stream and its events
        e2e_step()
    barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(k_e2e):
        e2e_step()
    torch.cuda.synchronize()
    barrier()
    e2e_ms = reduce_max((time.perf_counter() - t0) * 1e3 / k_e2e, ws)

    forms = {}
    if not args.no_forms:
        # plain form: one frame per launch, FP32; per-frame latency from events
        m1 = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight)
        s1 = make_step(m1, 1)
        for _ in range(args.warmup):
            s1()
        ms1 = timed(s1, max(3, args.steps // 2))
        lat = []
        m1.reset()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(n_frames)]
        for (a, b), f, d in zip(evs, w.frames, frames_dev):
            a.record()
            m1.integrate(f.sensor, f.T, d)
            b.record()
        torch.cuda.synchronize()
        lat = sorted(a.elapsed_time(b) for a, b in evs)
        forms["fp32_one_frame_per_launch"] = {
            "ms_per_step": ms1, "voxel_updates_per_s": ws * updates_per_step / (ms1 * 1e-3),
            "frames_per_s": ws * n_frames / (ms1 * 1e-3),
            "latency_ms": {"p50": lat[len(lat) // 2], "p99": lat[int(0.99 * (len(lat) - 1))]}}
        m1.close()
        # batched FP16 storage (precision pattern)
        m2 = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, storage=gt.STORAGE_FP16, **shape)
        s2 = make_step(m2, args.batch)
        for _ in range(args.warmup):
            s2()
        ms2 = timed(s2, args.steps)
        forms[f"fp16_batched_{args.batch}"] = {
            "ms_per_step": ms2, "voxel_updates_per_s": ws * updates_per_step / (ms2 * 1e-3),
            "frames_per_s": ws * n_frames / (ms2 * 1e-3)}
        m2.close()
        # occupancy layer (second update functor) over the same frames
        m3 = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight,
                        layer=gt.LAYER_OCCUPANCY)
        s3 = make_step(m3, args.batch)
        for _ in range(args.warmup):
            s3()
        ms3 = timed(s3, args.steps)
        forms[f"occupancy_batched_{args.batch}"] = {
            "ms_per_step": ms3, "voxel_updates_per_s": ws * m3.stats()["voxel_updates"] / (ms3 * 1e-3),
            "frames_per_s": ws * n_frames / (ms3 * 1e-3)}
        m3.close()
        # colour layer (Table I colour fusion): registered colour images
        colors = torch.from_numpy(synth.configs.room_colors(w).view(np.int32)).cuda()
        m4 = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, layer=gt.LAYER_COLOR)
        descs4 = [gt.frame_desc(0, f.sensor, f.T, d, colors[i])
                  for i, (f, d) in enumerate(zip(w.frames, frames_dev))]

        def s4():
            m4.reset()
            for s in range(0, n_frames, args.batch):
                gt.integrate_batch([m4.handle], descs4[s:s + args.batch])
        for _ in range(args.warmup):
            s4()
        ms4 = timed(s4, args.steps)
        forms[f"color_batched_{args.batch}"] = {
            "ms_per_step": ms4, "voxel_updates_per_s": ws * m4.stats()["voxel_updates"] / (ms4 * 1e-3),
            "frames_per_s": ws * n_frames / (ms4 * 1e-3)}
        m4.close()
        del colors
        # ESDF (Sec. IV-C) of the room map: built from all 300 frames, then
        # brought up to date after 10 more frames (incremental)
        m5 = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight)
        v32 = float(np.float32(w.voxel_size))
        # first calls on the empty map allocate the ESDF layer and the mesh
        # scratch and output (outside the timed calls); the step resets the map
        m5.esdf_update(v32, 1e-4, 64)
        m5.mesh(with_keys=False, cap=1 << 22)
        make_step(m5, args.batch)()

        def esdf_ms(fn):
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            torch.cuda.synchronize()
            return a.elapsed_time(b)
        full_ms = esdf_ms(lambda: m5.esdf_update(v32, 1e-4, 64))
        full_stats = m5.esdf_stats()
        descs5 = [gt.frame_desc(0, f.sensor, f.T, d) for f, d in zip(w.frames[:10], frames_dev[:10])]
        gt.integrate_batch([m5.handle], descs5)
        inc_ms = esdf_ms(lambda: m5.esdf_update(v32, 1e-4, 64))
        inc_stats = {k: v - full_stats[k] for k, v in m5.esdf_stats().items()}
        forms["esdf"] = {"blocks": m5.stats()["blocks"], "site_eps_m": v32, "max_dist_vox": 64,
                         "full_ms": full_ms, "full": full_stats,
                         "incremental_after_10_frames_ms": inc_ms, "incremental": inc_stats}
        # marching-cubes mesh of the same map: every block, then the blocks
        # changed by 10 more frames (and those whose cubes reach into them)
        mesh_full = [0]
        full_mesh_ms = esdf_ms(lambda: mesh_full.__setitem__(0, len(m5.mesh(with_keys=False, cap=1 << 22)[0])))
        m5.mesh(changed_only=True, with_keys=False, cap=1 << 22)  # consume the changes so far
        gt.integrate_batch([m5.handle], descs5)
        mesh_inc = [0]
        inc_mesh_ms = esdf_ms(lambda: mesh_inc.__setitem__(
            0, len(m5.mesh(changed_only=True, with_keys=False, cap=1 << 22)[0])))
        forms["mesh"] = {"full_ms": full_mesh_ms, "full_triangles": mesh_full[0],
                         "incremental_after_10_frames_ms": inc_mesh_ms,
                         "incremental_triangles": mesh_inc[0],
                         "note": "includes the output allocation and the count read-back"}
        m5.close()
        forms["fp32_batched_speedup_vs_one_frame"] = ms1 / ms
        forms["fp16_batched_speedup_vs_one_frame"] = ms1 / ms2
        # configs 4 and 5 at their stated sizes
        # one persistent launch per 32-frame sub-batch instead of two
        mf = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, launch_mode=gt.LAUNCH_FUSED)
        sf = make_step(mf, args.batch)
        for _ in range(args.warmup):
            sf()
        msf = timed(sf, args.steps)
        assert mf.stats()["voxel_updates"] == updates_per_step
        forms[f"fp32_fused_{args.batch}"] = {
            "ms_per_step": msf, "voxel_updates_per_s": ws * updates_per_step / (msf * 1e-3),
            "frames_per_s": ws * n_frames / (msf * 1e-3),
            "launch": "one cooperative launch per 32-frame sub-batch, sub-batches in sequence"}
        mf.close()
        if not args.no_rig:
            forms["rig_fp16"] = rig_form(args, torch, storage=gt.STORAGE_FP16)
            forms["rig_fp16_fused"] = rig_form(args, torch, storage=gt.STORAGE_FP16,
                                               launch_mode=gt.LAUNCH_FUSED)
            forms["rig_fixed16"] = rig_form(args, torch, storage=gt.STORAGE_FIXED16)
        if not args.no_serving:
            forms["serving_fp16"] = serving_form(args, torch, storage=gt.STORAGE_FP16)

    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(args.ref_frames)

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "storage": "fp32", "frames_per_call": args.batch,
                       "launch_shape": shape, "autotune": shape_timings,
                       "frames_per_launch": min(args.batch, 32),
                       "frames_per_step": n_frames, "voxel_updates_per_step": updates_per_step,
                       "l2": f"inputs {in_bytes / 1e6:.0f} MB resident in HBM (> 129 MB L2)",
                       "parallelism": f"replicas x{ws}"},
            "frames_per_s": fps,
            "roofline": {"bound": "hbm", "achieved": alloc_gbs, "peak": hbm_peak, "unit": "GB/s",
                         "frac": alloc_gbs / hbm_peak, "peak_source": peak_src,
                         "traffic": _traffic("patch_alloc_kernel"),
                         "kernel": "patch_alloc_kernel", "share_of_kernel_time": alloc_share,
                         "bytes_per_launch": alloc_bytes_per_launch,
                         "ms_per_launch": alloc_ms_per_launch,
                         "timing": "per-launch CUDA events inside the pipelined step",
                         "ms_per_launch_isolated": iso_alloc_ms,
                         "frac_isolated": alloc_bytes_per_launch / (iso_alloc_ms * 1e-3) / 1e9 / hbm_peak,
                         "note": "bytes: the depth images; issue and barriers bound the kernel"},
            "alloc_walk_equivalent": {"tops": alloc_ops_per_launch / (alloc_ms_per_launch * 1e-3) / 1e12,
                                      "tops_isolated": alloc_ops_per_launch / (iso_alloc_ms * 1e-3) / 1e12,
                                      "ops_per_launch": alloc_ops_per_launch,
                                      "segments_per_step": walk["segments"], "cells_per_step": walk["cells"],
                                      "note": "operations of walking every band segment, which the patch kernel "
                                              "avoids: comparable between versions, not with a peak"},
            # the integration is bound by issue (ALU), not by bytes: both views
            "roofline_integrate": {"bound": "alu", "achieved": integ_alu_achieved / 1e12,
                                   "peak": ALU_PEAK_OPS / 1e12, "unit": "Tops/s",
                                   "frac": integ_alu_achieved / ALU_PEAK_OPS,
                                   "traffic": _traffic("integrate_kernel"),
                                   "kernel": "integrate_kernel",
                                   "peak_source": "152 SMs x 128 lanes x 2070 MHz",
                                   "share_of_kernel_time": 1.0 - alloc_share,
                                   "ops_per_launch": integ_ops_per_launch,
                                   "block_frame_pairs_per_step": st["block_frame_pairs"],
                                   "ms_per_launch": integ_ms_per_launch,
                                   "timing": "per-launch CUDA events inside the pipelined step",
                                   "ms_per_launch_isolated": iso_integ / max(iso_calls, 1)},
            "roofline_integrate_hbm": {"bound": "hbm", "achieved": achieved, "peak": hbm_peak,
                                       "unit": "GB/s", "frac": achieved / hbm_peak,
                                       "traffic": _traffic("integrate_kernel"),
                                       "kernel": "integrate_kernel", "peak_source": peak_src,
                                       "bytes_per_launch": integ_bytes_per_launch,
                                       "ms_per_launch": integ_ms_per_launch,
                                   "timing": "per-launch CUDA events inside the pipelined step",
                                   "ms_per_launch_isolated": iso_integ / max(iso_calls, 1)},
            "kernel_ms_per_step": {"band_alloc": alloc_ms / args.steps,
                                   "integrate": integ_ms / args.steps,
                                   "note": "inside the pipelined step (the two kernels overlap)"},
            "kernel_ms_per_launch_isolated": {"band_alloc": iso_alloc / max(iso_calls, 1),
                                              "integrate": iso_integ / max(iso_calls, 1),
                                              "note": "one 32-frame sub-batch per call, kernels "
                                                      "not overlapped"},
            "e2e": {"value": ws * updates_per_step / (e2e_ms * 1e-3), "unit": UNIT,
                    "ms_per_step": e2e_ms, "h2d_bytes_per_step": in_bytes,
                    "d2h_bytes_per_step": 48,
                    "call": "integrate_batch_host (pinned host frames, copies overlapped) + map_stats"},
            "gpu_launches": args.steps * (1 + 2 * launches_per_step),
            "clocks": clk,
            "forms": forms,
            "cpu_baseline": cpu,
        }
        print(json.dumps(line), flush=True)
    m.close()
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def _setup_device():
    ws, rank, local = _dist()
    import torch
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    return ws, rank, local, torch


def _max_over_ranks(torch, ws, x):
    return reduce_max(x, ws)


def _hbm_view(bytes_per_launch: float, ms_per_launch: float, note: str):
    hbm, src = _peaks()
    gbs = bytes_per_launch / (ms_per_launch * 1e-3) / 1e9 if ms_per_launch > 0 else 0.0
    return {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
            "bytes_per_launch": bytes_per_launch, "ms_per_launch": ms_per_launch,
            "peak_source": src, "note": note}


def _block_bytes(storage: int) -> int:
    return 512 * (8 if storage == 0 else 4)


def rig_form(args, torch, storage: int = 1, graph_reps: int = 10, launch_mode: int = 0) -> dict:
    """Rig workload (one outdoor map at 0.05 m; per step four pinhole frames
    of 640x480 x2, 848x480, 1280x720 and one 1024x64 LiDAR scan in one
    integrate_batch call).  The whole sequence is captured once in a CUDA
    graph and replayed; the launch shape is picked by the autotuner.  Also
    the eager per-step latency and, from one eager run with per-launch
    events, the two kernels' times and the integrator's HBM view."""
    import paper_2311_00626_gb300 as gt
    from paper_2311_00626_gb300.serving import autotune
    import synth
    w = synth.config_rig(n_steps=args.rig_steps)
    n = len(w.frames)
    dev = [torch.from_numpy(f.depth).cuda() for f in w.frames]
    in_bytes = sum(int(d.numel()) * 4 for d in dev)
    steps = [list(range(s, s + 5)) for s in range(0, n, 5)]

    def make(cfg):
        m = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, storage=storage,
                       alloc_tile_h=cfg.get("alloc_tile_h", 0),
                       integrate_ctas_per_sm=cfg.get("integrate_ctas_per_sm", 0),
                       launch_mode=launch_mode)
        descs = [gt.frame_desc(0, w.frames[i].sensor, w.frames[i].T, dev[i]) for i in range(n)]

        def run():
            m.reset()
            for st in steps:
                gt.integrate_batch([m.handle], [descs[i] for i in st])
        return m, run, descs

    def time_cfg(cfg):
        m, run, _ = make(cfg)
        run()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        run()
        e1.record()
        torch.cuda.synchronize()
        m.close()
        return e0.elapsed_time(e1)

    cands = [{"alloc_tile_h": t, "integrate_ctas_per_sm": c} for t in (16, 32) for c in (0, 4, 6)]
    if launch_mode:  # one launch per step: only the tile height applies
        cands = [{"alloc_tile_h": t} for t in (16, 32)]
    best, timings = autotune(f"rig{args.rig_steps}s{storage}m{launch_mode}", time_cfg, cands, cache=False)
    m, run, descs = make(best)
    for _ in range(3):
        run()
    torch.cuda.synchronize()
    st = m.stats()
    updates = st["voxel_updates"]
    # eager per-step latency (one integrate_batch call per step)
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in steps]
    m.reset()
    for (a, b), s in zip(evs, steps):
        a.record()
        gt.integrate_batch([m.handle], [descs[i] for i in s])
        b.record()
    torch.cuda.synchronize()
    lat = sorted(a.elapsed_time(b) for a, b in evs)
    # per-kernel times from one eager run with events around every launch
    gt.map_timing(m.handle, True)
    run()
    alloc_ms, integ_ms, calls = gt.map_kernel_times(m.handle)
    gt.map_timing(m.handle, False)
    st = m.stats()
    # graph of the whole sequence, replayed
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        run()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        run()
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(graph_reps):
        g.replay()
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / graph_reps
    assert m.stats()["voxel_updates"] == updates, "non-deterministic update count"
    m.close()
    launches = len(steps)
    bytes_launch = ((2 * st["block_visits"] - st["blocks"]) * _block_bytes(storage) + in_bytes) / launches
    return {
        "storage": {0: "fp32", 1: "fp16", 2: "fixed16"}[storage],
        "launch": "fused: one launch per step" if launch_mode else "split: two launches per step",
        "ms_per_sequence": ms, "steps": len(steps), "frames": n,
        "voxel_updates_per_sequence": updates,
        "voxel_updates_per_s": updates / (ms * 1e-3), "frames_per_s": n / (ms * 1e-3),
        "rig_steps_per_s": len(steps) / (ms * 1e-3),
        "launch_shape": best, "autotune": timings,
        "eager_step_latency_ms": {"p50": lat[len(lat) // 2], "p99": lat[int(0.99 * (len(lat) - 1))]},
        "kernel_ms_per_launch": {"band_alloc": alloc_ms / max(calls, 1),
                                 "integrate": integ_ms / max(calls, 1)},
        "roofline_integrate_hbm": _hbm_view(
            bytes_launch, integ_ms / max(calls, 1),
            "algorithmic bytes: each listed block read and written once per launch "
            "(new blocks written only) plus the launch's images; eager launches"),
        "blocks": st["blocks"],
        "inputs": f"{in_bytes / 1e6:.0f} MB resident",
    }


def bench_rig(args):
    """`--workload rig`: the rig form alone as the JSON line."""
    ws, rank, local, torch = _setup_device()
    r = rig_form(args, torch, storage=1, graph_reps=args.steps)
    ms = _max_over_ranks(torch, ws, r["ms_per_sequence"])
    if rank == 0:
        print(json.dumps({
            "metric": METRIC, "value": ws * r["voxel_updates_per_sequence"] / (ms * 1e-3), "unit": UNIT,
            "n_gpus": ws, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": f"rig outdoor 40x40x5 m, {r['steps']} steps x (4 pinhole + 1 LiDAR), "
                                   "voxel 0.05 m, FP16 storage, CUDA graph of the whole sequence",
                       "launch_shape": r["launch_shape"]},
            "frames_per_s": ws * r["frames"] / (ms * 1e-3), "rig": r,
            "gpu_launches": args.steps * (1 + 2 * r["steps"]),
        }), flush=True)


# Algorithmic bytes of the derived layers (FP32 TSDF blocks of 4096 B, ESDF
# state blocks of 2048 B): what each stage must read and write at least.
TSDF_BLOCK_B = 512 * 8
ESDF_BLOCK_B = 512 * 4
ESDF_FACES_B = 6 * 64 * 4
TRI_POS_B = 9 * 4


def esdf_bytes(marked: int, swept: int, pulled: int) -> int:
    """Marking reads a changed block's TSDF and reads and writes its state;
    a sweep reads and writes a block's state; a face exchange reads the
    block's state and its six neighbours' facing faces."""
    return (marked * (TSDF_BLOCK_B + 2 * ESDF_BLOCK_B) + swept * 2 * ESDF_BLOCK_B
            + pulled * (ESDF_BLOCK_B + ESDF_FACES_B))


def mesh_bytes(blocks: int, tris: int) -> int:
    """Meshing reads each listed block's TSDF once and writes each triangle's
    three vertex positions."""
    return blocks * TSDF_BLOCK_B + tris * TRI_POS_B


def bench_layers(args):
    """Derived layers of the room map (300 frames, 2 cm, FP32): every step
    resets the map and integrates the 300 frames (untimed), then times the
    ESDF from scratch (Sec. IV-C), the ESDF brought up to date after 10 more
    frames, the marching-cubes mesh of every block (Sec. IV-B) and the mesh
    of the blocks those 10 frames changed.  Each call is timed with CUDA
    events on the stream it runs on, host-side convergence checks and the
    triangle-count read-back included."""
    import numpy as np
    ws, rank, local, torch = _setup_device()
    import paper_2311_00626_gb300 as gt
    import synth
    w = synth.config_room(n_frames=300)
    dev = torch.from_numpy(np.stack([f.depth for f in w.frames])).cuda()
    descs = [gt.frame_desc(0, f.sensor, f.T, dev[i]) for i, f in enumerate(w.frames)]
    v32 = float(np.float32(w.voxel_size))
    m = gt.TsdfMap(w.voxel_size, w.truncation_voxels, w.max_weight, storage=gt.STORAGE_FP32)
    # the first calls allocate the ESDF layer and the mesh scratch
    m.esdf_update(v32, 1e-4, 64)
    m.mesh(with_keys=False, cap=1 << 22)
    cap = 1 << 22

    def timed_call(fn):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        out = fn()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b), out

    def step():
        r = {}
        m.reset()
        gt.integrate_batch([m.handle], descs)
        blocks = m.stats()["blocks"]
        e0 = m.esdf_stats()
        r["esdf_full_ms"], _ = timed_call(lambda: m.esdf_update(v32, 1e-4, 64))
        e1 = m.esdf_stats()
        v0 = m.stats()["block_visits"]
        gt.integrate_batch([m.handle], descs[:10])
        changed = m.stats()["block_visits"] - v0
        r["esdf_inc_ms"], _ = timed_call(lambda: m.esdf_update(v32, 1e-4, 64))
        e2 = m.esdf_stats()
        r["mesh_full_ms"], t_full = timed_call(lambda: len(m.mesh(with_keys=False, cap=cap)[0]))
        m.mesh(changed_only=True, with_keys=False, cap=cap)  # consume the changes so far
        gt.integrate_batch([m.handle], descs[10:20])
        r["mesh_inc_ms"], t_inc = timed_call(
            lambda: len(m.mesh(changed_only=True, with_keys=False, cap=cap)[0]))
        r["blocks"], r["changed"], r["tris_full"], r["tris_inc"] = blocks, changed, t_full, t_inc
        r["full"] = {k: e1[k] - e0[k] for k in e1}
        r["inc"] = {k: e2[k] - e1[k] for k in e2}
        return r

    for _ in range(args.warmup):
        step()
    runs = [step() for _ in range(args.steps)]
    last = runs[-1]
    for r in runs:  # the work is the same every step
        assert (r["blocks"], r["tris_full"], r["full"]) == (last["blocks"], last["tris_full"], last["full"])

    def mean(k):
        return _max_over_ranks(torch, ws, float(np.mean([r[k] for r in runs])))
    t = {k: mean(k) for k in ("esdf_full_ms", "esdf_inc_ms", "mesh_full_ms", "mesh_inc_ms")}
    hbm, hbm_src = _peaks()

    def roof(nbytes, ms):
        gbs = nbytes / (ms * 1e-3) / 1e9
        return {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                "bytes": nbytes, "peak_source": hbm_src}

    esdf_launches = 3  # mark, clear, and every lowering iteration in one
    # the mesh lists every block whose cubes reach into a changed block, up
    # to eight per changed block; the changed blocks bound it from below
    rl = {
        "esdf_full": roof(esdf_bytes(last["blocks"], last["full"]["swept"], last["full"]["pulled"]),
                          t["esdf_full_ms"]),
        "esdf_incremental": roof(esdf_bytes(last["changed"], last["inc"]["swept"], last["inc"]["pulled"]),
                                 t["esdf_inc_ms"]),
        "mesh_full": roof(mesh_bytes(last["blocks"], last["tris_full"]), t["mesh_full_ms"]),
        "mesh_incremental": roof(mesh_bytes(last["changed"], last["tris_inc"]), t["mesh_inc_ms"]),
    }
    ms = sum(t.values())
    if rank == 0:
        print(json.dumps({
            "metric": "ESDF and mesh update time of the room map", "value": ms, "unit": "ms",
            "n_gpus": ws, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int32/f32",
            "data": "synthetic",
            "config": {"workload": "room 10x10x3 m, 300 frames 640x480 f=525, voxel 0.02 m, FP32 TSDF; "
                                   "ESDF max distance 64 voxels, sites |D| <= 1 voxel; then 10 more frames",
                       "blocks": last["blocks"], "blocks_changed_by_10_frames": last["changed"],
                       "l2": "TSDF 83 MB and ESDF state 42 MB: largely L2-resident (129 MB)"},
            "ms": t, "triangles": {"full": last["tris_full"], "incremental": last["tris_inc"]},
            "esdf": {"full": last["full"], "incremental": last["inc"]},
            "roofline": rl,
            "gpu_launches": args.steps * (2 * esdf_launches + 2 * 2),
        }), flush=True)
    m.close()


def _serving_requests(torch, seconds: float, pool: int):
    """Config-5 request stream: 16 maps, Poisson 30 Hz per map for `seconds`
    of simulated time; each request's depth is rendered from the map's
    seeded room at one of `pool` poses of its path (the poses cycle), by the
    sensor drawn for it.  Renders run on a thread pool (the C renderer
    releases the interpreter lock)."""
    import numpy as np
    from concurrent.futures import ThreadPoolExecutor
    import synth
    from paper_2311_00626_gb300.serving import Request
    from synth.configs import (ROOM_NOISE, SERVING_SENSORS, config_serving_maps, render_frame,
                               serving_arrivals)
    cfg = config_serving_maps(16)
    arrivals = serving_arrivals(16, 30.0, seconds)
    poses = [synth.trajectory(c["seed"], c["prims"], pool) for c in cfg]
    count = [0] * 16
    keys = []
    for t, mid, si in arrivals:
        keys.append((t, mid, si, count[mid] % pool))
        count[mid] += 1

    def pose(mid, k, si):
        T = poses[mid][k]
        if SERVING_SENSORS[si]["kind"] == "lidar":
            T = T.copy()
            T[:3, :3] = np.eye(3)  # LiDAR mounted level, z up
        return T

    def render(key):
        mid, k, si = key
        s = SERVING_SENSORS[si]
        d = render_frame(cfg[mid]["prims"], s, pose(mid, k, si),
                         ROOM_NOISE if s["kind"] == "pinhole" else {"sigma": 0.02},
                         cfg[mid]["seed"], k * 4 + si)
        return key, torch.from_numpy(d).pin_memory()

    distinct = sorted({(mid, k, si) for _, mid, si, k in keys})
    with ThreadPoolExecutor(max(1, min(16, os.cpu_count() or 1))) as ex:
        cache = dict(ex.map(render, distinct))
    reqs = [Request(i, mid, SERVING_SENSORS[si], pose(mid, k, si), cache[(mid, k, si)], t)
            for i, (t, mid, si, k) in enumerate(keys)]
    return cfg, reqs, len(distinct)


def serving_form(args, torch, storage: int = 1) -> dict:
    """Serving workload (config 5): 16 device-resident maps (voxel 0.02 /
    0.05 / 0.1 m), Poisson arrivals at 30 Hz per map for --serve-seconds of
    simulated time of 320x240 / 640x480 / 1280x720 depth or 1024x64 LiDAR
    frames; continuous batching with admission by staging footprint.
    Unpaced throughput (every request available at once; median of three
    runs), paced p50 / p99 latency (arrivals follow the wall clock), and from
    one more unpaced run with per-launch events the kernels' times and the
    integrator's HBM view over all maps."""
    import paper_2311_00626_gb300 as gt
    from paper_2311_00626_gb300.serving import Request, Server
    cfg, reqs, distinct = _serving_requests(torch, args.serve_seconds, args.serve_pool)
    # the maps persist across runs (reset in between): per-map set-up
    # (sensor tables, the copy stream) stays outside the timed runs
    maps = [gt.TsdfMap(c["voxel_size"], c["truncation_voxels"], c["max_weight"], storage=storage,
                       max_blocks=args.serve_max_blocks)
            for c in cfg]
    in_bytes = sum(r.nbytes for r in reqs)

    def serve(paced, timing=False):
        for m in maps:
            m.reset()
            if timing:
                gt.map_timing(m.handle, True)
        rs = [Request(r.rid, r.map_id, r.sensor, r.T, r.depth, r.arrival if paced else 0.0)
              for r in reqs]
        srv = Server(maps, staging_bytes=512 << 20, max_frames=32)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        done = srv.run(rs, paced=paced)
        wall = time.perf_counter() - t0
        sts = [m.stats() for m in maps]
        out = {"wall_s": wall, "voxel_updates": sum(s["voxel_updates"] for s in sts),
               "launches": srv.launches, **Server.latency_stats(done)}
        if timing:
            a = i = 0.0
            calls = 0
            for m in maps:
                am, im, c = gt.map_kernel_times(m.handle)
                gt.map_timing(m.handle, False)
                a, i, calls = a + am, i + im, calls + c
            out["kernel_ms"] = {"band_alloc": a, "integrate": i, "launches": calls}
            out["block_visits"] = sum(s["block_visits"] for s in sts)
            out["blocks"] = sum(s["blocks"] for s in sts)
        return out

    serve(False)  # warm-up
    runs = sorted((serve(False) for _ in range(3)), key=lambda r: r["wall_s"])
    unpaced = runs[1]
    unpaced["wall_s_runs"] = [r["wall_s"] for r in runs]
    tm = serve(False, timing=True)
    paced = serve(True)
    for m in maps:
        m.close()
    k = tm["kernel_ms"]
    bytes_launch = ((2 * tm["block_visits"] - tm["blocks"]) * _block_bytes(storage) + in_bytes) / max(k["launches"], 1)
    return {
        "storage": {0: "fp32", 1: "fp16", 2: "fixed16"}[storage],
        "simulated_s": args.serve_seconds, "frames": len(reqs), "distinct_images": distinct,
        "poses_per_map": args.serve_pool,
        "voxel_updates_per_s": unpaced["voxel_updates"] / unpaced["wall_s"],
        "frames_per_s": len(reqs) / unpaced["wall_s"],
        "unpaced": unpaced, "paced": paced,
        "latency_ms": {"p50": paced["p50_ms"], "p99": paced["p99_ms"]},
        "kernel_ms_per_launch": {"band_alloc": k["band_alloc"] / max(k["launches"], 1),
                                 "integrate": k["integrate"] / max(k["launches"], 1)},
        "roofline_integrate_hbm": _hbm_view(
            bytes_launch, k["integrate"] / max(k["launches"], 1),
            "algorithmic bytes: each listed block read and written once per launch "
            "(new blocks written only) plus the launch's images; one unpaced run"),
        "map_bytes": tm["blocks"] * _block_bytes(storage),
        "inputs": f"{in_bytes / 1e9:.2f} GB of requests, {distinct} distinct pinned images",
    }


def bench_serving(args):
    """`--workload serving`: the serving form alone as the JSON line."""
    ws, rank, local, torch = _setup_device()
    r = serving_form(args, torch)
    if rank == 0:
        print(json.dumps({
            "metric": METRIC, "value": ws * r["voxel_updates_per_s"], "unit": UNIT, "n_gpus": ws,
            "steps": 3, "warmup": 1, "ms_per_step": r["unpaced"]["wall_s"] * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": f"serving: 16 maps, Poisson 30 Hz per map for {args.serve_seconds} s "
                                   f"({r['frames']} frames), mixed sensors, FP16, "
                                   f"{args.serve_pool} poses per map"},
            "frames_per_s": ws * r["frames_per_s"], "serving": r,
        }), flush=True)


if __name__ == "__main__":
    main()
