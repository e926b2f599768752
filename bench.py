"""Benchmark of the LiteVoxel rasterizer training step on GB300.

One step = the whole hot path over one view of the Mip-NeRF-360-shaped
synthetic scene (2M voxels, levels 6-12, 1237x822, FP32 storage):
stats reset, forward (binning, pair sort, composite with w_max), LF-weighted
loss, backward (composite + SH), w_max unpack, depth-quantile pruning and
priority subdivision (into separate output buffers, so every step does the
same work).  The metric is forward+backward throughput in Mpix/s.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

With N > 1 (torchrun, one process per GPU) every rank runs an independent
replica of the step on its own view; nothing is exchanged between ranks.
--impl reference times the CPU oracle (the FP64/FP32 reference written from
the paper) on a bounded sample of the same workload on the host cores.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "fwd+bwd Mpix/s at 1 GB300, batched/mixed vs plain FP32; % HBM roofline"
UNIT = "Mpix/s"
W_IMG, H_IMG = 1237, 822
WORKLOAD = ("360-scene 2M voxels (levels 6-12, background shell r 12-16, opaque surfaces), 1 view 1237x822, "
            "FP32 storage")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--seed", type=int, default=0)
    # a fixed composite schedule instead of the autotuner's choice (for profiler runs, whose
    # distorted timings would steer the autotuner elsewhere): tile edge and 0 / 1 for persistent
    ap.add_argument("--tile", type=int, choices=[8, 16, 32], default=None)
    ap.add_argument("--persistent", type=int, choices=[0, 1], default=None)
    ap.add_argument("--batch", type=int, choices=[32, 64, 128], default=32)
    return ap.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def max_over_ranks(x: float, world: int, device=None) -> float:
    """Largest value of x over all ranks (the step time of the slowest replica)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def tuned_schedule(scene, cams):
    """Tile size and composite schedule from the library's autotuner (lv_autotune: every
    tile size with and without persistent warps, forward + backward timed with CUDA
    events on this scene and these views), as a user of the library would pick them."""
    import torch

    from paper_2511_02510_gb300 import litevoxel as L
    from paper_2511_02510_gb300.raster import RasterContext
    vox = scene.voxels()
    probe = RasterContext(cams, scene.n)
    probe.fit_capacity(vox)  # the pair capacity the default tile needs
    cap = 2 * probe.pair_capacity  # smaller tiles cut voxels into more pairs
    base = L.make_opts()
    ws = torch.empty(L.lv_autotune_workspace_size(scene.n, probe.cams_arr, len(cams), base, cap),
                     dtype=torch.uint8, device="cuda")
    best, ms = L.lv_autotune(vox, probe.cams_arr, len(cams), base, cap, 3, ws)
    del ws, probe
    torch.cuda.empty_cache()
    return int(best.tile), bool(best.flags & L.LV_FLAG_PERSISTENT), int(best.batch), ms


TUNE_TILES, TUNE_BATCHES = (8, 16, 32), (32, 64, 128)


def step_batch_candidates(tile, persistent, batch, tune_ms, within=0.03):
    """Batches of the tuner's tile and schedule whose forward + backward time (lv_autotune's
    ms_out, index 6 t + 3 p + b) lies within `within` of the fastest: the tuner's pick first.
    (All of them while the batch changes no launch, so the step does not choose among them.)"""
    if not tune_ms or tile not in TUNE_TILES:
        return [batch]
    t, p = TUNE_TILES.index(tile), 1 if persistent else 0
    ms = {b: tune_ms[6 * t + 3 * p + i] for i, b in enumerate(TUNE_BATCHES)}
    best = min(v for v in ms.values() if v > 0) if any(v > 0 for v in ms.values()) else None
    if best is None:
        return [batch]
    return [batch] + [b for b in TUNE_BATCHES if b != batch and ms[b] > 0 and ms[b] <= (1 + within) * best]


def camera_for(rank: int):
    from paper_2511_02510_gb300 import synth
    return synth.orbit_camera(W_IMG, H_IMG, 60.0, 3.0, 37.0 + 45.0 * rank, 15.0)


# ---------------------------------------------------------------------------- GPU workload
class Workload:
    """Device-resident training state for one view and the buffers of one step."""

    def __init__(self, scene_np, cam, gt_np, density_dtype=None, sh_dtype=None, t_iter=450.0, tuned=False,
                 schedule=None):
        import torch

        from paper_2511_02510_gb300 import litevoxel as L
        from paper_2511_02510_gb300.raster import RasterContext, Scene

        self.torch, self.L = torch, L
        dd = density_dtype or torch.float32
        sd = sh_dtype or torch.float32
        n = int(scene_np["geom"].shape[0])
        self.n = n
        # the voxel arrays hold room for the step's growth: the topology change is written in place
        # (top 5 % split: at most n + 7 * 0.05 n rows)
        cap = n + 7 * (n * 50000 // 1000000) + 16
        self.cap = cap
        src = Scene.from_numpy(scene_np, "cuda", dd, sd)
        big = [torch.empty((cap,) + tuple(t.shape[1:]), dtype=t.dtype, device="cuda")
               for t in (src.geom, src.level, src.density, src.sh)]
        for b, t in zip(big, (src.geom, src.level, src.density, src.sh)):
            b[:n].copy_(t)
        del src
        self.cap_arrays = big  # geometry, level, corners, SH with room for the growth
        self.scene = Scene(big[0][:n], big[1][:n], big[2][:n], big[3][:n])
        self.cams = [cam]
        self.tile, self.persistent, self.batch, self.tune_ms = 16, False, 32, None
        if schedule is not None:
            self.tile, self.persistent, self.batch = schedule
        elif tuned:
            self.tile, self.persistent, self.batch, self.tune_ms = tuned_schedule(self.scene, self.cams)
        self.rctx = RasterContext(self.cams, n, tile=self.tile, batch=self.batch, persistent=self.persistent)
        # the step's backward composite is the persistent one, on all but 64 SMs, which it leaves to the
        # pruning and selection kernels that the four-stream step runs beside it (graph-replayed step:
        # 0.811 ms with the backward on 88 SMs, 0.814 on 80, 0.819 on 72, 0.823 on 96, 0.830 on 120);
        # the forward composite runs alone, by the schedule the tuner picks
        self.persistent_sms = max(1, torch.cuda.get_device_properties(0).multi_processor_count - 64)
        self.bwd_opts = L.make_opts(self.tile, self.batch, persistent=True, persistent_sms=self.persistent_sms)
        self.vox = self.scene.voxels()
        self.rctx.fit_capacity(self.vox)
        self.npix = self.rctx.n_pix
        dev = "cuda"
        self.gt = torch.as_tensor(gt_np).to(dev).contiguous()
        self.gt_host = torch.as_tensor(gt_np).pin_memory()
        self.loss = torch.zeros(1, dtype=torch.float32, device=dev)
        self.loss_host = torch.zeros(1, dtype=torch.float32).pin_memory()
        self.dL = torch.empty((self.npix, 3), dtype=torch.float32, device=dev)
        self.d_dens = torch.empty((n, 8), dtype=torch.float32, device=dev)
        self.d_sh = torch.empty((n, 48), dtype=torch.float32, device=dev)
        self.w_max = torch.empty(n, dtype=torch.float32, device=dev)
        self.w_arg = torch.empty(n, dtype=torch.int64, device=dev)
        self.t_iter = t_iter
        # LF loss (Eq. 7-10, 18), mid-ramp
        self.lfp = L.lv_lf_params()
        self.lfp.eps, self.lfp.gamma_max, self.lfp.t0, self.lfp.t1, self.lfp.pctl_ppm = 1e-3, 0.6, 300.0, 600.0, 990000
        self.lf_ws = torch.empty(L.lv_lf_workspace_size([W_IMG], [H_IMG]), dtype=torch.uint8, device=dev)
        # pruning (q = 5 %, 16 bins, EMA decay 0.9, cap 1 %)
        self.pp = L.lv_prune_params()
        self.pp.n_bins, self.pp.q_ppm, self.pp.ema_alpha, self.pp.m_low, self.pp.m_high = 16, 50000, 0.1, 0.3, 0.7
        self.pp.cap_ppm, self.pp.lo_ppm, self.pp.hi_ppm = 10000, 50000, 950000
        self.pr_ws = torch.empty(L.lv_prune_workspace_size(n, self.pp), dtype=torch.uint8, device=dev)
        # EMA state of a voxel set that training has been pruning: every voxel just above m_low, so
        # one out-vote moves it out and the cap (guard iii) decides how many go, from the first step
        self.ema_cap = torch.full((cap,), 0.32, dtype=torch.float32, device=dev)
        self.state_cap = torch.ones(cap, dtype=torch.uint8, device=dev)
        self.ema, self.state = self.ema_cap[:n], self.state_cap[:n]
        self.ema0, self.state0 = self.ema.clone(), self.state.clone()
        self.pmask = torch.empty(n, dtype=torch.uint8, device=dev)
        self.n_pruned = torch.zeros(1, dtype=torch.int64, device=dev)
        # subdivision (kappa 1, beta 0.2, top 5 %), written in place
        self.sp = L.lv_subdiv_params()
        self.sp.kappa, self.sp.beta, self.sp.top_ppm, self.sp.l_max = 1.0, 0.2, 50000, 16
        self.sp.budget, self.sp.lo_ppm, self.sp.hi_ppm = 1 << 40, 50000, 950000
        self.sd_ws = torch.empty(L.lv_subdivide_workspace_size(n, self.sp), dtype=torch.uint8, device=dev)
        self.selected = torch.empty(n, dtype=torch.uint8, device=dev)
        self.n_new = torch.zeros(1, dtype=torch.int64, device=dev)
        self.status = torch.zeros(1, dtype=torch.int32, device=dev)
        # optimizer moments and EMA state carried through the topology change, updated in place
        self.aux_arrays = [torch.zeros((cap, 8), dtype=torch.float32, device=dev),
                           torch.zeros((cap, 8), dtype=torch.float32, device=dev),
                           torch.zeros((cap, 48), dtype=torch.float32, device=dev),
                           torch.zeros((cap, 48), dtype=torch.float32, device=dev), self.ema_cap, self.state_cap]
        fills = [0, 0, 0, 0, int(np.array([1.0], np.float32).view(np.uint32)[0]), 1]
        self.aux = []
        for t, f in zip(self.aux_arrays, fills):
            a = L.lv_aux_array()
            a.in_, a.out = t.data_ptr(), t.data_ptr()
            a.width = 1 if t.dim() == 1 else t.shape[1]
            a.elem_bytes = t.element_size()
            a.fill = f
            self.aux.append(a)
        self.restore_idx = None

    # stage boundaries, for the per-kernel breakdown
    STAGES = ["reset", "forward", "loss", "backward", "sh_backward", "unpack", "prune", "subdivide_select",
              "subdivide_inplace", "restore"]

    def _state_arrays(self):
        """The per-voxel arrays the next step reads that an in-place topology change overwrites below
        row n: geometry, level, corners and SH (the optimizer moments are only written by the step,
        and the EMA and hysteresis state is restored whole)."""
        sc = self.scene
        return [sc.geom, sc.level, sc.density, sc.sh]

    def prepare_restore(self, pristine):
        """After one step taken from the state `pristine` (clones of _state_arrays() from before it):
        note the rows that step's topology change overwrote (split parents and filled holes: the rows
        selected or pruned), keep their original contents, and put the whole state back.  Every step
        takes the same decisions from the same state, so restore() returns the state after each step."""
        torch = self.torch
        idx = torch.nonzero((self.selected != 0) | (self.pmask != 0)).flatten()
        self.restore_idx = idx
        self.restore_saved = [p.index_select(0, idx) for p in pristine]
        for arr, p in zip(self._state_arrays(), pristine):
            arr.copy_(p)
        self.ema.copy_(self.ema0)
        self.state.copy_(self.state0)

    def restore(self):
        """Put back the rows the step's in-place topology change overwrote and the pruning state, so
        the next step starts from the same scene (inside the timed region: it is extra work), in
        one launch of the library's row scatter."""
        if self.restore_idx is None:
            return
        items = [(arr, saved, self.restore_idx) for arr, saved in zip(self._state_arrays(), self.restore_saved)]
        items += [(self.ema, self.ema0, None), (self.state, self.state0, None)]
        self.L.lv_rows_scatter(items)

    def step(self, ev=None):
        L, r = self.L, self.rctx

        def mark(i):
            if ev is not None:
                ev[i].record()

        mark(0)
        r.reset_stats()
        self.d_dens.zero_()
        mark(1)
        r.forward(self.vox, stats=True)
        mark(2)
        L.lv_lf_weighted_loss(r.rgb, self.gt, [W_IMG], [H_IMG], self.t_iter, self.lfp, self.loss, self.dL, self.lf_ws)
        mark(3)
        L.lv_rasterize_backward(self.vox, r.cams_arr, r.n_views, r.opts, r.fwd_struct(False), r.workspace,
                                r.pair_capacity, self.dL, None, None, self.d_dens, None, True, r.status)
        mark(4)
        L.lv_sh_backward(self.vox, r.cams_arr, r.n_views, r.opts, r.workspace, r.pair_capacity, self.d_sh, False)
        mark(5)
        L.lv_unpack_wmax(r.wmax_packed, self.w_max, self.w_arg)
        mark(6)
        L.lv_prune_depth_quantile(self.w_max, r.seen, r.z_min, self.ema, self.state, self.pp, self.pmask,
                                  self.n_pruned, self.pr_ws)
        mark(7)
        L.lv_subdivide_select(self.vox, r.delta_min, r.z_min, self.w_max, r.seen, self.pmask, self.sp, self.cap,
                              self.selected, self.n_new, self.sd_ws, self.status)
        mark(8)
        L.lv_subdivide_apply_inplace(self.vox, self.cap, self.sp, self.aux, self.sd_ws)
        mark(9)
        self.restore()
        mark(10)

    def step_concurrent(self, ev=None):
        """The same work as step(), in three streams.  The LF weight map depends on the ground
        truth only, and pruning and the subdivision selection on the forward statistics only, so
        they run beside the forward and the backward respectively (side streams at high priority,
        joined by events): the depth bins of the pruning start as soon as the forward has binned
        the voxels (its statistics event), the rest once w_max is out.  The LF loss's gradient is
        fused into the backward composite (which waits for the weights), its value is finished
        after it.  The SH backward, which reads the forward's workspace and not the voxel
        arrays, runs beside the topology change and the restore.  The in-place topology
        change runs last, alone, then the restore.  ev: {"composite" | "backward" | "apply":
        (start, end)} timing events (external, so that they time graph replays)."""
        torch, L, r = self.torch, self.L, self.rctx
        if not hasattr(self, "_side"):
            hi = torch.cuda.Stream.priority_range()[1]
            # the SH backward gets a stream of normal priority: its many blocks must not hold up the
            # pruning and selection chain, which ends last
            self._side = (torch.cuda.Stream(priority=hi), torch.cuda.Stream(priority=hi), torch.cuda.Stream())
            self._evs = [torch.cuda.Event() for _ in range(7)]
            self._evs[4].record()  # the statistics event must exist before the library records it
        sw, sb, sl = self._side
        e_start, e_w, e_fwd, e_b, e_stats, e_bwd, e_sh = self._evs
        main = torch.cuda.current_stream()
        e_start.record(main)
        sw.wait_event(e_start)
        with torch.cuda.stream(sw):
            self.d_dens.zero_()
            L.lv_lf_weights(self.gt, [W_IMG], [H_IMG], self.t_iter, self.lfp, self.lf_ws)
            e_w.record(sw)
        r.reset_stats()
        r.forward(self.vox, stats=True, stats_event=e_stats, composite_event=ev["composite"][0] if ev else None)
        if ev:
            ev["composite"][1].record(main)
        e_fwd.record(main)
        sb.wait_event(e_stats)
        with torch.cuda.stream(sb):
            L.lv_prune_bins(r.seen, r.z_min, self.pp, self.pr_ws)
        sb.wait_event(e_fwd)
        with torch.cuda.stream(sb):
            L.lv_unpack_wmax(r.wmax_packed, self.w_max, self.w_arg)
            L.lv_prune_finish(self.w_max, r.seen, r.z_min, self.ema, self.state, self.pp, self.pmask,
                              self.n_pruned, self.pr_ws)
            L.lv_subdivide_select(self.vox, r.delta_min, r.z_min, self.w_max, r.seen, self.pmask, self.sp,
                                  self.cap, self.selected, self.n_new, self.sd_ws, self.status)
            e_b.record(sb)
        if ev:
            ev["backward"][0].record(main)
        # the LF loss's gradient is fused into the backward composite, which waits for the weights (e_w)
        L.lv_rasterize_backward(self.vox, r.cams_arr, r.n_views, self.bwd_opts,
                                r.fwd_struct(False, lf=(self.gt, self.lf_ws, self.dL, e_w)), r.workspace,
                                r.pair_capacity, None, None, None, self.d_dens, None, True, r.status)
        if ev:
            ev["backward"][1].record(main)
        L.lv_lf_loss_finish([W_IMG], [H_IMG], self.loss, self.lf_ws)
        # the SH backward reads only the workspace, so it runs beside the in-place topology change;
        # it waits for the selection too, whose memory-bound chain it would otherwise slow down
        e_bwd.record(main)
        sl.wait_event(e_bwd)
        sl.wait_event(e_b)
        with torch.cuda.stream(sl):
            L.lv_sh_backward(self.vox, r.cams_arr, r.n_views, r.opts, r.workspace, r.pair_capacity, self.d_sh,
                             False)
            e_sh.record(sl)
        main.wait_event(e_b)
        if ev:
            ev["apply"][0].record(main)
        L.lv_subdivide_apply_inplace(self.vox, self.cap, self.sp, self.aux, self.sd_ws)
        if ev:
            ev["apply"][1].record(main)
        self.restore()
        main.wait_event(e_sh)

    def e2e_step(self):
        """The same step through the public API with host buffers: the step's ground-truth
        image is copied from pinned host memory and the loss is read back."""
        self.gt.copy_(self.gt_host, non_blocking=True)
        self.step()
        self.loss_host.copy_(self.loss, non_blocking=True)
        self.torch.cuda.current_stream().synchronize()
        return float(self.loss_host[0])

    def counters(self):
        pairs, slots = self.rctx.counters()
        return {"pairs": pairs, "visible_slots": slots, "n_pruned": int(self.n_pruned.item()),
                "n_new": int(self.n_new.item()), "status": int(self.status.item() | self.rctx.status.item()),
                "samples": int(self.rctx.n_samples.to(self.torch.int64).sum().item()),
                "split": int(self.selected.to(self.torch.int64).sum().item())}

    def row_bytes(self):
        """Bytes of one voxel's state rows: geometry, level, corners, SH and the auxiliary arrays."""
        b = 16 + 1 + 8 * self.scene.density.element_size() + 48 * self.scene.sh.element_size()
        return b + sum(t[0].numel() * t.element_size() for t in self.aux_arrays)


# ---------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        # the raw samples (summarised into the JSON line); LV_BENCH_OUT chooses the folder
        out_dir = os.environ.get("LV_BENCH_OUT") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"clocks_rank{gpu_index}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"], stdout=self.f,
                                         stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.3)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        with open(self.path) as f:
            return clock_summary(f)


CLOCK_REASONS = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")


def clock_summary(lines):
    """Median SM clock, the highest max clock and the throttle reasons seen active, from nvidia-smi CSV
    lines in ``ClockSampler.FIELDS`` order (no header, no units); lines that do not parse are skipped.
    None without a sample."""
    sm, mx, reasons = [], [], set()
    for line in lines:
        parts = [p.strip() for p in line.split(",")]
        if len(parts) < 9:
            continue
        try:
            clock, max_clock = float(parts[1]), float(parts[2])
        except ValueError:
            continue
        sm.append(clock)
        mx.append(max_clock)
        for name, v in zip(CLOCK_REASONS, parts[5:9]):
            if v.lower() == "active":
                reasons.add(name)
    if not sm:
        return None
    return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons), "samples": len(sm)}


# ---------------------------------------------------------------------------- roofline
def dram_traffic(kernel):
    """DRAM bytes per launch of ``kernel`` from the committed ncu capture, or None
    when none was taken or the kernel's source changed since it was: the hash
    covers the region of the source file that holds the kernel and its device
    helpers (``source_region``: first and end marker), else the whole file."""
    tp = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(tp):
        return None
    rec = json.load(open(tp)).get(kernel)
    if not rec:
        return None
    with open(os.path.join(ROOT, rec["source"]), encoding="utf-8") as f:
        text = f.read()
    if rec.get("source_region"):
        first, end = rec["source_region"]
        i = text.find(first)
        j = text.find(end, i) if i >= 0 else -1
        if i < 0 or j < 0:
            return None
        text = text[i:j]
    if hashlib.sha256(text.encode("utf-8")).hexdigest() != rec["source_sha256"]:
        return None
    return int(rec["dram_bytes_per_launch"])


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


# FP32 operations of one composited sample (an FMA counts 2, a min/max/compare or MUFU op 1):
# chord 18, midpoint + trilinear 30, opacity 8, accumulation 12 -> forward 68;
# backward: chord 18, midpoint + trilinear 30, transmittance and weight 14,
# dL/dsigma 12, corner and colour gradients 28 -> 102.
FLOPS_PER_SAMPLE = {"forward_composite": 68, "backward_composite": 102}
SMS, FP32_LANES = 152, 128


def alu_peak_tflops(sm_mhz):
    """FP32 peak of the GB300 at the given SM clock: 152 SMs x 128 lanes x 2 (FMA)."""
    return SMS * FP32_LANES * 2 * sm_mhz * 1e6 / 1e12


def stage_work(n, slots, pairs, npix, tiles, samples, split, pruned, row, parent_row):
    """Algorithmic bytes and FP32 operations of every stage of one step (FP32 storage): what each
    stage must read and write at least once.  Rasterizer stages a1-a7 as the scope table of the
    method's hot path counts them (N voxels, N_v visible slots, P (tile, slot) pairs, Npx pixels,
    S composited samples); then the LF loss (Eq. 7-10), w_max unpack, pruning (Eq. 11-12),
    the subdivision selection (Eq. 13-16) and the in-place topology change."""
    N, Nv, P, Npx, S, k, h = n, slots, pairs, npix, samples, split, pruned
    st = {
        "a1_preprocess": (N * 16 + Nv * (192 + 28), 0),
        "a2_scan_emit": (Nv * 8 + P * 12, 0),
        "a3_sort": (P * 24, 0),
        "a4_tile_ranges": (P * 8 + tiles * 8, 0),
        "a5_forward_composite": (P * (4 + 64) + Npx * 24 + P * 8, S * FLOPS_PER_SAMPLE["forward_composite"]),
        "a6_backward_composite": (P * (4 + 64) + Npx * 40 + P * 11 * 8, S * FLOPS_PER_SAMPLE["backward_composite"]),
        "a7_sh_backward": (Nv * (12 + 192 + 192), 0),
        "lf_loss": (Npx * 36, 0),                               # gt and rgb read, dL/drgb written
        "reset_and_unpack": (N * 17 + N * 20, 0),               # statistics reset; packed w_max -> w_max, argmax
        "prune": (N * 20, 0),                                   # w_max, seen, z, m, s read; m, s, mask written
        "subdivide_select": (N * 32, 0),                        # geometry, level, delta, z, u, seen, mask; selected
        "subdivide_inplace": (k * parent_row + 8 * k * row + N + 4 * h, 0),
    }
    return {name: {"bytes": int(b), "flops": int(f)} for name, (b, f) in st.items()}


def step_roofline(work, ms_step, hbm_gbs, fp32_tflops):
    """Sum over stages of max(bytes / HBM peak, flops / FP32 peak), against the measured step time."""
    total = 0.0
    out = {}
    for name, w in work.items():
        t_mem = w["bytes"] / (hbm_gbs * 1e9) * 1e3
        t_alu = w["flops"] / (fp32_tflops * 1e12) * 1e3
        out[name] = {"bytes": w["bytes"], "flops": w["flops"], "bound_ms": max(t_mem, t_alu),
                     "bound": "hbm" if t_mem >= t_alu else "alu"}
        total += max(t_mem, t_alu)
    return {"stages": out, "sum_bound_ms": total, "ms_per_step": ms_step, "frac": total / ms_step}


# ---------------------------------------------------------------------------- CPU baseline (oracle)
def oracle_step_time(scene_np, cam, gt_np):
    """Wall time of one step of the oracle on the whole 1237x822 view: FP64 render (Eq. 1-5), LF loss
    (Eq. 7-10), reverse pass, FP32 binning statistics, pruning (Eq. 11-12) from the same initial EMA
    state as the GPU step, and subdivision (Eq. 13-16) on all voxels."""
    from oracle import oracle as O
    n = scene_np["geom"].shape[0]
    t0 = time.perf_counter()
    r = O.render(scene_np, [cam])
    t1 = time.perf_counter()
    lf = O.lf_loss(r["rgb"], gt_np.astype(np.float64).reshape(-1, 3), [(W_IMG, H_IMG)],
                   gamma=O.lf_gamma(450.0, 300.0, 600.0, 0.6))
    O.render_backward(scene_np, [cam], lf["dL_drgb"])
    t2 = time.perf_counter()
    st = O.pairs(scene_np, [cam])
    w = r["w_max"].astype(np.float32)
    pr = O.prune(w, st["seen"], st["z_min"], np.full(n, 0.32, np.float32), np.ones(n, np.uint8))
    O.subdivide(scene_np, st["delta_min"], st["z_min"], w, st["seen"], prune_mask=pr["mask"])
    t3 = time.perf_counter()
    sample = (f"the whole step on the whole 1237x822 view: render {t1 - t0:.2f} s, LF loss + backward "
              f"{t2 - t1:.2f} s, binning statistics + prune + subdivide on all {n} voxels {t3 - t2:.2f} s")
    return t3 - t0, sample


def cpu_baseline(scene_np, cam, gt_np):
    from oracle import oracle as O
    step, sample = oracle_step_time(scene_np, cam, gt_np)
    return {"value": (W_IMG * H_IMG) / step / 1e6, "unit": UNIT, "cores": O.num_threads(), "kind": "oracle",
            "sample": sample, "seconds": step}


# ---------------------------------------------------------------------------- arms
def run_reference(args, rank):
    if rank != 0:
        return
    from oracle import oracle as O
    from paper_2511_02510_gb300 import synth
    O.build()
    scene_np = synth.scene_360(seed=args.seed)
    cam = camera_for(0)
    gt_np = synth.random_image(W_IMG, H_IMG, seed=1)
    times = []
    sample = ""
    for i in range(args.warmup + args.steps):
        st, sample = oracle_step_time(scene_np, cam, gt_np)
        if i >= args.warmup:
            times.append(st)
    ms = 1e3 * float(np.mean(times))
    value = (W_IMG * H_IMG) / (ms / 1e3) / 1e6
    print(json.dumps({"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
                      "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
                      "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                      "config": {"workload": WORKLOAD, "global_batch": 1, "seq_len": None,
                                 "parallelism": "cpu oracle"},
                      "cpu_baseline": {"value": value, "unit": UNIT, "cores": O.num_threads(), "kind": "oracle",
                                       "sample": sample + " (measured anew each step)"},
                      "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}),
          flush=True)


def run_stress(torch, synth, steps=50, budget=12_000_000):
    """The growth-budget stress workload: ~10M voxels, 8 views of 1600x1060, FP16 corners and BF16
    SH, each step forward + LF loss (gamma ramp 0 -> 1 over the run) + backward + prune + subdivide
    under the voxel budget, the scene growing in place of the old one (ping-pong buffers)."""
    from paper_2511_02510_gb300 import litevoxel as L
    from paper_2511_02510_gb300.raster import RasterContext
    dev = "cuda"
    sc = synth.scene_stress()
    n0 = int(sc["geom"].shape[0])
    W, H, V = 1600, 1060, 8
    cams = [synth.orbit_camera(W, H, 60.0, 4.0, 45.0 * i, 15.0) for i in range(V)]
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    base_mem = torch.cuda.memory_allocated()
    cap = budget + 8

    def arrays():
        return {"geom": torch.empty((cap, 4), device=dev), "level": torch.empty(cap, dtype=torch.uint8, device=dev),
                "density": torch.empty((cap, 8), dtype=torch.float16, device=dev),
                "sh": torch.empty((cap, 48), dtype=torch.bfloat16, device=dev),
                "ema": torch.empty(cap, device=dev), "state": torch.empty(cap, dtype=torch.uint8, device=dev)}

    bufs = [arrays(), arrays()]
    a = bufs[0]
    a["geom"][:n0].copy_(torch.as_tensor(sc["geom"]))
    a["level"][:n0].copy_(torch.as_tensor(sc["level"]))
    a["density"][:n0].copy_(torch.as_tensor(sc["density"]).half())
    a["sh"][:n0].copy_(torch.as_tensor(sc["sh"]).bfloat16())
    a["ema"][:n0].fill_(1.0)
    a["state"][:n0].fill_(1)
    del sc
    ctx = RasterContext(cams, cap)
    vox0 = L.make_voxels(a["geom"], a["density"], a["sh"], a["level"])
    vox0.n = n0
    pairs = ctx.fit_capacity(vox0, headroom=2.0)
    gt = torch.from_numpy(np.concatenate([synth.smooth_image(W, H, seed=i) for i in range(V)])).to(dev)
    lp = L.lv_lf_params()
    lp.eps, lp.gamma_max, lp.t0, lp.t1, lp.pctl_ppm = 1e-3, 1.0, 0.3 * steps, 0.6 * steps, 990000
    lf_ws = torch.empty(L.lv_lf_workspace_size([W] * V, [H] * V), dtype=torch.uint8, device=dev)
    loss = torch.zeros(V, device=dev)
    dL = torch.empty((ctx.n_pix, 3), device=dev)
    d_dens = torch.empty((cap, 8), device=dev)
    d_sh = torch.empty((cap, 48), device=dev)
    w_max = torch.empty(cap, device=dev)
    pp = L.lv_prune_params()
    pp.n_bins, pp.q_ppm, pp.ema_alpha, pp.m_low, pp.m_high, pp.cap_ppm = 16, 50000, 0.1, 0.3, 0.7, 10000
    pp.lo_ppm, pp.hi_ppm = 50000, 950000
    pws = torch.empty(L.lv_prune_workspace_size(cap, pp), dtype=torch.uint8, device=dev)
    mask = torch.empty(cap, dtype=torch.uint8, device=dev)
    npr = torch.zeros(1, dtype=torch.int64, device=dev)
    sp = L.lv_subdiv_params()
    sp.kappa, sp.beta, sp.top_ppm, sp.l_max, sp.budget, sp.lo_ppm, sp.hi_ppm = 1.0, 0.2, 50000, 16, budget, 50000, 950000
    sws = torch.empty(L.lv_subdivide_workspace_size(cap, sp), dtype=torch.uint8, device=dev)
    sel = torch.empty(cap, dtype=torch.uint8, device=dev)
    nn = torch.zeros(1, dtype=torch.int64, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    n = n0
    counts = []
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for it in range(steps):
        a, b = bufs[it % 2], bufs[1 - it % 2]
        vox = L.make_voxels(a["geom"], a["density"], a["sh"], a["level"])
        vox.n = n
        ctx.reset_stats()
        ctx.forward(vox)
        L.lv_lf_weighted_loss(ctx.rgb, gt, [W] * V, [H] * V, float(it), lp, loss, dL, lf_ws)
        L.lv_rasterize_backward(vox, ctx.cams_arr, ctx.n_views, ctx.opts, ctx.fwd_struct(False), ctx.workspace,
                                ctx.pair_capacity, dL, None, None, d_dens[:n], d_sh[:n], False, ctx.status)
        L.lv_unpack_wmax(ctx.wmax_packed[:n], w_max[:n])
        L.lv_prune_depth_quantile(w_max[:n], ctx.seen[:n], ctx.z_min[:n], a["ema"][:n], a["state"][:n], pp,
                                  mask[:n], npr, pws)
        aux = []
        for key, fill in (("ema", 1.0), ("state", 1)):
            x = L.lv_aux_array()
            x.in_, x.out, x.width = a[key].data_ptr(), b[key].data_ptr(), 1
            x.elem_bytes = a[key].element_size()
            x.fill = int(np.array([fill], np.float32 if key == "ema" else np.uint8).view(
                np.uint32 if key == "ema" else np.uint8)[0])
            aux.append(x)
        vout = L.make_voxels(b["geom"], b["density"], b["sh"], b["level"])
        vout.n = cap
        L.lv_subdivide_priority(vox, ctx.delta_min[:n], ctx.z_min[:n], w_max[:n], ctx.seen[:n], mask[:n], sp, aux,
                                vout, sel[:n], nn, sws, status)
        n = int(nn.item())  # the next step's voxel count (one host read per step)
        counts.append(n)
    e1.record()
    torch.cuda.synchronize()
    ctx.check()
    if int(status.item()) != 0:
        raise RuntimeError(f"stress: device status {int(status.item())}")
    ms = e0.elapsed_time(e1) / steps
    return {"value": ctx.n_pix / (ms / 1e3) / 1e6, "unit": UNIT, "ms_per_step": ms, "steps": steps,
            "views": V, "pixels": ctx.n_pix, "voxels_start": n0, "voxels_end": counts[-1],
            "voxels_max": max(counts), "budget": budget, "pairs_first_step": int(pairs),
            "peak_vram_gb": (torch.cuda.max_memory_allocated() - base_mem) / 1e9,
            "step": "forward + LF loss (gamma ramp 0 -> 1) + backward (corners and SH) + prune + subdivide, "
                    "growing under the budget",
            "density_dtype": "float16", "sh_dtype": "bfloat16"}


def run_variant(torch, synth, kind, scene_np, steps=10, warmup=3):
    """Batched / mixed-precision / semi-transparent variants measured beside the plain path (same GPU)."""
    from paper_2511_02510_gb300 import litevoxel as L
    from paper_2511_02510_gb300.raster import RasterContext, Scene
    if kind == "batched16_fp32":
        sc = scene_np
        cams = synth.uneven_views(16, seed=2)
        dd, sd = torch.float32, torch.float32
    elif kind == "batched8_mixed":  # the 2M scene, 8 views of 980x545, BF16 SH + FP16 corners
        sc = scene_np
        cams = [synth.orbit_camera(980, 545, 60.0, 3.0, 45.0 * i, 15.0) for i in range(8)]
        dd, sd = torch.float16, torch.bfloat16
    elif kind in ("plain_fp32", "exact_segment_fp32", "persistent_fp32"):  # the plain view (variants)
        sc = scene_np
        cams = [camera_for(0)]
        dd, sd = torch.float32, torch.float32
    else:  # semi_transparent_fp32: the plain view of the same octree with peak density 10 per unit
        sc = synth.scene_360(opaque=False)
        cams = [camera_for(0)]
        dd, sd = torch.float32, torch.float32
    scene = Scene.from_numpy(sc, "cuda", dd, sd)
    tile, persistent, batch = 16, kind == "persistent_fp32", 32
    if kind in ("plain_fp32", "batched16_fp32", "batched8_mixed"):  # the autotuned schedule, as the bench step
        tile, persistent, batch, _ = tuned_schedule(scene, cams)
    ctx = RasterContext(cams, scene.n, tile=tile, batch=batch, exact_segment=(kind == "exact_segment_fp32"),
                        persistent=persistent)
    vox = scene.voxels()
    ctx.fit_capacity(vox)
    g = torch.randn((ctx.n_pix, 3), device="cuda") * 1e-3
    dd_ = torch.empty((scene.n, 8), device="cuda")
    ds_ = torch.empty((scene.n, 48), device="cuda")

    def step():
        ctx.reset_stats()
        ctx.forward(vox)
        ctx.backward(vox, g, d_density=dd_, d_sh=ds_)

    from paper_2511_02510_gb300.raster import CapturedStep
    for _ in range(warmup):
        step()
    torch.cuda.synchronize()
    graph = CapturedStep(step)  # one launch per step, as the plain path is timed
    for _ in range(warmup):
        graph()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        graph()
    e1.record()
    torch.cuda.synchronize()
    ctx.check()
    ms = e0.elapsed_time(e1) / steps
    return {"value": ctx.n_pix / (ms / 1e3) / 1e6, "unit": UNIT, "ms_per_step": ms, "views": len(cams),
            "pixels": ctx.n_pix, "tile": tile, "batch": batch, "persistent": persistent, "density_dtype": str(dd).split(".")[-1], "sh_dtype": str(sd).split(".")[-1],
            "step": "stats reset + forward + backward (composite + SH), replayed as one CUDA graph"}


def _time_ms(torch, fn, reps, warm=3):
    """Mean device time of fn() over reps launches (CUDA events on the current stream)."""
    for _ in range(warm):
        fn()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(reps):
        fn()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def run_next_rows(torch, L, wl, reps, hbm_peak):
    """The rows beyond the per-step hot path, each timed on its own on the same scene and view:
    the Adam update with the fused density TV gradient, the transmittance-concentration loss, and
    the pruning guards (keep-halo with the edge map, annealed q_b, running percentiles)."""
    n, dev = wl.n, "cuda"
    out = {}
    # Adam + TV: in place on copies of the parameters, FP32 moments
    dens, sh = wl.scene.density.clone(), wl.scene.sh.clone()
    md, vd = torch.zeros((n, 8), device=dev), torch.zeros((n, 8), device=dev)
    ms, vs = torch.zeros((n, 48), device=dev), torch.zeros((n, 48), device=dev)
    tws = torch.empty(L.lv_train_workspace_size(), dtype=torch.uint8, device=dev)
    tvl = torch.zeros(1, device=dev)
    p = L.lv_adam_params()
    p.lr_density, p.lr_sh, p.beta1, p.beta2, p.eps, p.step, p.tv_weight = 1e-2, 2.5e-3, 0.9, 0.999, 1e-15, 10, 1e-4
    ms_adam = _time_ms(torch, lambda: L.lv_adam_voxels(dens, sh, wl.d_dens, wl.d_sh, md, vd, ms, vs, p, tws,
                                                       tv_loss=tvl), reps)
    row = 7 * 8 * 4 + 7 * 48 * 4            # param, grad, m, v read; param, m, v written (FP32)
    gbs = n * row / (ms_adam / 1e3) / 1e9
    out["adam_tv"] = {"ms": ms_adam, "bound": "hbm", "achieved": gbs, "peak": hbm_peak, "unit": "GB/s",
                      "frac": gbs / hbm_peak, "bytes_per_voxel": row, "voxels": n,
                      "kernels": "k_adam_density (fused L_tv gradient) + k_adam_flat (SH)"}
    # transmittance concentration on the view's final T
    dT = torch.empty(wl.npix, device=dev)
    tcl = torch.zeros(1, device=dev)
    ms_tc = _time_ms(torch, lambda: L.lv_transmittance_loss(wl.rctx.T, 0.01, tcl, dT, tws), reps)
    gbs = wl.npix * 8 / (ms_tc / 1e3) / 1e9
    out["transmittance_loss"] = {"ms": ms_tc, "bound": "hbm", "achieved": gbs, "peak": hbm_peak, "unit": "GB/s",
                                 "frac": gbs / hbm_peak, "pixels": wl.npix}
    # pruning with every guard on: edge map from the loss, per-voxel gather, keep-halo, q_b, running pct
    edge_map = torch.empty(wl.npix, device=dev)
    edge = torch.empty(n, device=dev)
    pct = torch.full((2,), float("nan"), device=dev)
    ema, state = wl.ema.clone(), wl.state.clone()
    pg = L.lv_prune_params()
    for f, _ in L.lv_prune_params._fields_[:8]:
        setattr(pg, f, getattr(wl.pp, f))
    pg.anneal, pg.anneal_ppm, pg.relax_ppm = 1, L.lv_prune_anneal_ppm(wl.t_iter, 0.0, 900.0), 200000
    pg.halo_small, pg.halo_w, pg.halo_edge = 0.5, 0.5, 0.5
    pg.geom, pg.delta, pg.edge = wl.scene.geom.data_ptr(), wl.rctx.delta_min.data_ptr(), edge.data_ptr()
    pg.pct_ema, pg.pct_state = 0.1, pct.data_ptr()
    lf_edge = L.lv_lf_params()
    for f, _ in L.lv_lf_params._fields_[:5]:
        setattr(lf_edge, f, getattr(wl.lfp, f))
    lf_edge.edge_out = edge_map.data_ptr()

    def plain():
        L.lv_lf_weighted_loss(wl.rctx.rgb, wl.gt, [W_IMG], [H_IMG], wl.t_iter, wl.lfp, wl.loss, wl.dL, wl.lf_ws)
        L.lv_prune_depth_quantile(wl.w_max, wl.rctx.seen, wl.rctx.z_min, ema, state, wl.pp, wl.pmask,
                                  wl.n_pruned, wl.pr_ws)

    def guarded():
        L.lv_lf_weighted_loss(wl.rctx.rgb, wl.gt, [W_IMG], [H_IMG], wl.t_iter, lf_edge, wl.loss, wl.dL, wl.lf_ws)
        L.lv_gather_edge(wl.w_arg, edge_map, edge)
        L.lv_prune_depth_quantile(wl.w_max, wl.rctx.seen, wl.rctx.z_min, ema, state, pg, wl.pmask, wl.n_pruned,
                                  wl.pr_ws)

    ms_plain = _time_ms(torch, plain, reps)
    ms_guard = _time_ms(torch, guarded, reps)
    # shared grid-vertex densities: index build, then forward + backward + vertex-gradient scatter
    from paper_2511_02510_gb300.raster import RasterContext
    unit = float(wl.scene.geom[:, 3].min())
    vidx = torch.empty((n, 8), dtype=torch.int32, device=dev)
    nvt = torch.zeros(1, dtype=torch.int64, device=dev)
    ms_index = _time_ms(torch, lambda: L.lv_build_vertex_index(wl.scene.geom, unit, vidx, nvt), 3, warm=1)
    n_vert = int(nvt.item())
    vsum, vcnt = torch.zeros(n_vert, device=dev), torch.zeros(n_vert, device=dev)
    L.lv_vertex_scatter_add(vidx, wl.scene.density, vsum, vcnt)
    vdens = vsum / vcnt.clamp_min(1.0)
    vvox = L.make_voxels(wl.scene.geom, vdens, wl.scene.sh, vidx=vidx)
    vctx = RasterContext(wl.cams, n)
    vctx.fit_capacity(vvox)
    gvert = torch.zeros(n_vert, device=dev)
    dcorner = torch.empty((n, 8), device=dev)
    dsh = torch.empty((n, 48), device=dev)

    def vstep():
        vctx.reset_stats()
        vctx.forward(vvox)
        vctx.backward(vvox, wl.dL, d_density=dcorner, d_sh=dsh)
        gvert.zero_()
        L.lv_vertex_scatter_add(vidx, dcorner, gvert)

    ms_vstep = _time_ms(torch, vstep, reps)
    out["vertex_densities"] = {"vertices": n_vert, "ms_build_index": ms_index,
                               "ms_fwd_bwd_scatter": ms_vstep, "mpix_s": wl.npix / (ms_vstep / 1e3) / 1e6,
                               "step": "stats reset + forward + backward (composite + SH) + vertex scatter"}
    out["prune_guards"] = {"ms_loss_and_prune": ms_plain, "ms_loss_and_prune_with_guards": ms_guard,
                           "overhead_ms": ms_guard - ms_plain,
                           "guards": "keep-halo (size + edge), annealed relaxed q_b, running percentiles"}
    return out


def run_ours(args, rank, world, local):
    import torch
    import torch.distributed as dist

    from paper_2511_02510_gb300 import build as B
    from paper_2511_02510_gb300 import litevoxel as L
    from paper_2511_02510_gb300 import synth

    B.build()
    L.load()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    def barrier():
        if world > 1:
            dist.barrier()

    scene_np = synth.scene_360(seed=args.seed)
    cam = camera_for(rank)
    gt_np = synth.random_image(W_IMG, H_IMG, seed=1 + rank)
    fixed = ((args.tile, bool(args.persistent), args.batch) if args.tile is not None and args.persistent is not None
             else None)
    wl = Workload(scene_np, cam, gt_np, tuned=True, schedule=fixed)
    # one step from the initial state shows which rows the in-place topology change overwrites; every
    # later step restores them (and the pruning state) at its end, so all steps do the same work
    pristine = [a.clone() for a in wl._state_arrays()]
    wl.step()
    torch.cuda.synchronize()
    first = wl.counters()
    wl.prepare_restore(pristine)
    del pristine
    torch.cuda.empty_cache()
    for _ in range(max(3, args.warmup)):
        wl.step()
    torch.cuda.synchronize()
    cnt = wl.counters()
    if cnt["status"] != 0:
        raise RuntimeError(f"device status {cnt['status']} during warm-up")
    if any(cnt[k] != first[k] for k in ("n_pruned", "n_new", "split", "pairs")):
        raise RuntimeError(f"the restored state does not repeat the first step: {first} vs {cnt}")
    from paper_2511_02510_gb300.raster import CapturedStep

    # ---- per-stage breakdown: K eager steps with an event at every stage boundary
    K = args.steps
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(len(Workload.STAGES) + 1)] for _ in range(K)]
    launches0 = L.launch_count()
    wl.step()
    launches_per_step = L.launch_count() - launches0
    torch.cuda.synchronize()
    for k in range(K):
        wl.step(evs[k])
    torch.cuda.synchronize()
    # medians over the K steps: one step that the host delays (a launch held up by the scheduler)
    # must not move a stage's time
    stage_ms = {s: float(np.median([evs[k][i].elapsed_time(evs[k][i + 1]) for k in range(K)]))
                for i, s in enumerate(Workload.STAGES)}
    eager_ms = float(np.median([evs[k][0].elapsed_time(evs[k][-1]) for k in range(K)]))

    # ---- timed region: K replays of the step captured in one CUDA graph
    graph_step = CapturedStep(wl.step_concurrent)
    for _ in range(max(3, args.warmup)):
        graph_step()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clk = ClockSampler(local)
    barrier()
    torch.cuda.synchronize()
    clk.start()
    time.sleep(0.2)
    e0.record()
    for k in range(K):
        graph_step()
    e1.record()
    torch.cuda.synchronize()
    barrier()
    clocks = clk.stop()
    launches = launches_per_step * K
    ms = e0.elapsed_time(e1) / K
    ms_max = max_over_ranks(ms, world, "cuda")
    value = world * wl.npix / (ms_max / 1e3) / 1e6

    # ---- end to end through the API with host buffers: every step copies its ground-truth image from
    # pinned host memory to the device and reads its loss back into pinned host memory, and the host
    # reads every step's loss.  Like a training loop that logs its loss asynchronously, the host reads
    # step k's loss while step k+1 runs, and step k+1's image uploads (on a copy stream) while step k
    # computes; two device image buffers and two host loss buffers, one captured graph per pair.
    gt_bufs = (wl.gt, torch.empty_like(wl.gt))
    loss_bufs = (wl.loss_host, torch.zeros_like(wl.loss_host).pin_memory())

    def e2e_body():
        wl.step_concurrent()
        wl.loss_host.copy_(wl.loss, non_blocking=True)

    e2e_graphs = []
    for buf, lbuf in zip(gt_bufs, loss_bufs):
        wl.gt, wl.loss_host = buf, lbuf
        buf.copy_(wl.gt_host)
        e2e_graphs.append(CapturedStep(e2e_body))
    wl.gt, wl.loss_host = gt_bufs[0], loss_bufs[0]
    main_s = torch.cuda.current_stream()
    copy_s = torch.cuda.Stream()
    ev_ready = [torch.cuda.Event(), torch.cuda.Event()]
    ev_used = [torch.cuda.Event(), torch.cuda.Event()]
    losses = []

    def e2e_run(steps):
        with torch.cuda.stream(copy_s):
            gt_bufs[0].copy_(wl.gt_host, non_blocking=True)
            ev_ready[0].record(copy_s)
        for k in range(steps):
            b = k % 2
            if k + 1 < steps:  # upload the next step's image while this one computes
                nb = 1 - b
                with torch.cuda.stream(copy_s):
                    if k >= 1:
                        copy_s.wait_event(ev_used[nb])
                    gt_bufs[nb].copy_(wl.gt_host, non_blocking=True)
                    ev_ready[nb].record(copy_s)
            main_s.wait_event(ev_ready[b])
            e2e_graphs[b]()
            ev_used[b].record(main_s)
            if k >= 1:  # the previous step's loss, read while this step runs
                ev_used[1 - b].synchronize()
                losses.append(float(loss_bufs[1 - b][0]))
        ev_used[(steps - 1) % 2].synchronize()
        losses.append(float(loss_bufs[(steps - 1) % 2][0]))
        copy_s.synchronize()

    e2e_run(3)
    barrier()
    t0 = time.perf_counter()
    e2e_run(K)
    e2e_s = (time.perf_counter() - t0) / K
    e2e_val = world * wl.npix / max_over_ranks(e2e_s, world, "cuda") / 1e6

    # kernels inside graph replays of the same step: timing events captured around the composite
    # (from the forward's composite event), the backward composite and the in-place topology change,
    # read after each of K more replays
    kernel_ms = {}
    try:
        # external: recorded as event nodes of the graph (rather than turned into a stream dependency)
        marks = {k: (torch.cuda.Event(enable_timing=True, external=True),
                     torch.cuda.Event(enable_timing=True, external=True)) for k in ("composite", "backward", "apply")}
        for a, b in marks.values():
            a.record()
            b.record()
        g_marked = CapturedStep(lambda: wl.step_concurrent(ev=marks))
        samples = {k: [] for k in marks}
        for _ in range(K):
            g_marked()
            torch.cuda.synchronize()
            for k, (a, b) in marks.items():
                samples[k].append(a.elapsed_time(b))
        kernel_ms = {k: float(np.median(v)) for k, v in samples.items()}
        del g_marked
    except Exception as e:  # event nodes in a graph: fall back to the eager stage times if refused
        print(f"graph-timed kernels unavailable: {e!r}", file=sys.stderr)
        kernel_ms = {}

    # the out-of-place form of the same topology change (lv_subdivide_apply: every survivor copied to
    # new arrays), on the last step's selection, for comparison
    oop_ms = None
    try:
        cap = wl.cap
        og = [torch.empty((cap,) + tuple(t.shape[1:]), dtype=t.dtype, device="cuda")
              for t in (wl.scene.geom, wl.scene.level, wl.scene.density, wl.scene.sh)]
        vout = L.make_voxels(og[0], og[2], og[3], og[1])
        vout.n = cap
        aux_o, keep_o = [], []
        for a, t in zip(wl.aux, wl.aux_arrays):
            o = torch.empty_like(t)
            x = L.lv_aux_array()
            x.in_, x.out, x.width, x.elem_bytes, x.fill = t.data_ptr(), o.data_ptr(), a.width, a.elem_bytes, a.fill
            aux_o.append(x)
            keep_o.append(o)
        oop_ms = _time_ms(torch, lambda: L.lv_subdivide_apply(wl.vox, wl.sp, aux_o, vout, wl.sd_ws), K)
        del og, vout, aux_o, keep_o
        torch.cuda.empty_cache()
    except Exception as e:
        print(f"out-of-place comparison unavailable: {e!r}", file=sys.stderr)

    cnt = wl.counters()
    if any(cnt[k] != first[k] for k in ("n_pruned", "n_new", "split", "pairs")):
        raise RuntimeError(f"the timed steps did not repeat the first step: {first} vs {cnt}")
    if rank == 0:
        hbm_peak, peak_src = peaks()
        sm_mhz = clocks["sm_mhz"] if clocks else 2070.0
        fp32_peak = alu_peak_tflops(sm_mhz)
        row = wl.row_bytes()
        parent_row = 16 + 1 + 8 * wl.scene.density.element_size() + 48 * wl.scene.sh.element_size()
        tiles = sum(((c["width"] + wl.tile - 1) // wl.tile) * ((c["height"] + wl.tile - 1) // wl.tile)
                    for c in wl.cams)
        work = stage_work(wl.n, cnt["visible_slots"], cnt["pairs"], wl.npix, tiles, cnt["samples"], cnt["split"],
                          cnt["n_pruned"], row, parent_row)
        # the kernels timed inside graph replays; their algorithmic bytes and FP32 operations
        names = {"composite": ("k_fwd (front-to-back composite, Eq. 2-5)", "a5_forward_composite"),
                 "backward": ("k_bwd (back-to-front composite, reverse of Eq. 2-4)", "a6_backward_composite"),
                 "apply": ("k_ip_children + k_ip_tail (in-place topology change, Sec. IV-D)", "subdivide_inplace")}
        fallback = {"composite": None, "backward": stage_ms["backward"], "apply": stage_ms["subdivide_inplace"]}
        kernels = {}
        for key, (label, stage) in names.items():
            t = kernel_ms.get(key) or fallback[key]
            if not t:
                continue
            w = work[stage]
            gbs = w["bytes"] / (t / 1e3) / 1e9
            tfl = w["flops"] / (t / 1e3) / 1e12
            kernels[key] = {"kernel": label, "ms": t, "algorithmic_bytes": w["bytes"], "flops": w["flops"],
                            "achieved_gbs": gbs, "hbm_frac": gbs / hbm_peak, "achieved_tflops": tfl,
                            "fp32_frac": tfl / fp32_peak,
                            "timing": "graph replays (event nodes, median of K)" if kernel_ms.get(key)
                                      else "eager stage events (median of K)"}
            if key == "apply":
                kernels[key]["note"] = ("runs beside the SH backward (another stream), with which it shares "
                                        "HBM; the topology change alone takes about 0.10 ms")
        dom = max(kernels, key=lambda k_: kernels[k_]["ms"])
        d = kernels[dom]
        traffic_key = {"composite": "k_fwd", "backward": "k_bwd", "apply": "k_ip_children"}[dom]
        roofline = {"bound": "hbm", "kernel": d["kernel"], "achieved": d["achieved_gbs"], "peak": hbm_peak,
                    "unit": "GB/s", "frac": d["hbm_frac"], "traffic": dram_traffic(traffic_key),
                    "peak_source": peak_src, "algorithmic_bytes": d["algorithmic_bytes"], "kernel_ms": d["ms"],
                    "kernel_timing": d["timing"], "kernels": kernels,
                    "fp32_peak_tflops": fp32_peak,
                    "fp32_peak_source": f"derived: 152 SMs x 128 FP32 lanes x 2 x {sm_mhz:.0f} MHz",
                    "step_level": step_roofline(work, ms_max, hbm_peak, fp32_peak)}
        out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K, "warmup": args.warmup,
               "ms_per_step": ms_max, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
               "dtype": "f32", "data": "synthetic",
               "config": {"workload": WORKLOAD, "model": "LiteVoxel sparse-voxel tile rasterizer",
                          "global_batch": world, "seq_len": None, "parallelism": f"replicas x{world}",
                          "voxels": wl.n, "pixels_per_rank": wl.npix, "pairs": cnt["pairs"],
                          "visible_slots": cnt["visible_slots"], "tile": wl.tile, "batch": wl.batch,
                          "schedule": ("forward: " + ("persistent warps" if wl.persistent else "a warp per strip") +
                                       f" (autotuned); backward: persistent warps on {wl.persistent_sms} SMs"),
                          "autotune_ms": wl.tune_ms,
                          "l2": "inputs larger than L2 (scene arrays 480 MB, per-step outputs > 600 MB)"},
               "roofline": roofline,
               "stages_ms": stage_ms, "eager_ms_per_step": eager_ms,
               "timing": "device time of K replays of the step captured in one CUDA graph (CUDA events); the "
                         "step runs on four streams (LF weights beside the forward; the backward composite fuses "
                         "the LF loss's gradient; pruning and the subdivision selection beside the backward; the SH "
                         "backward beside the in-place topology change); every step ends by restoring the rows "
                         "its topology change overwrote and the pruning state (one lv_rows_scatter launch, "
                         "inside the timed region), so that all steps do the same work; stages_ms from K eager "
                         "one-stream steps with an event at every stage boundary",
               "e2e": {"value": e2e_val, "unit": UNIT, "h2d_bytes_per_step": int(wl.gt_host.numel() * 4),
                       "d2h_bytes_per_step": 4,
                       "how": "host wall clock of K steps through the API: each step's ground-truth image is "
                              "copied from pinned host memory (on a copy stream, overlapping the previous step) and "
                              "its loss is copied back to pinned host memory and read by the host while the next "
                              "step runs"},
               "gpu_launches": int(launches),
               "restore": {"rows": int(wl.restore_idx.numel()), "launches_per_step": 1,
                           "what": "one lv_rows_scatter launch: the overwritten rows of the geometry, level, "
                                   "corner and SH arrays put back, and full copies of the EMA and hysteresis "
                                   "state, inside the timed region (extra work, not part of the method)"},
               "topology_change": {"inplace_ms": kernels.get("apply", {}).get("ms"),
                                   "out_of_place_ms": oop_ms,
                                   "inplace_bytes": work["subdivide_inplace"]["bytes"],
                                   "out_of_place_bytes": (wl.n - cnt["n_pruned"] - cnt["split"]) * row * 2
                                   + 8 * cnt["split"] * row + cnt["split"] * parent_row},
               "clocks": clocks,
               "step_counters": cnt}
        if not args.no_variants:
            try:
                out["variants"] = {k: run_variant(torch, synth, k, scene_np)
                                   for k in ("batched16_fp32", "batched8_mixed", "semi_transparent_fp32",
                                             "exact_segment_fp32", "persistent_fp32")}
                out["variants"]["stress_10M_growth"] = run_stress(torch, synth)
                out["variants"]["plain_fp32"] = run_variant(torch, synth, "plain_fp32", scene_np)
                plain = out["variants"]["plain_fp32"]["value"]
                out["variants"]["ratios_vs_plain_fp32"] = {
                    k: out["variants"][k]["value"] / plain for k in ("batched16_fp32", "batched8_mixed")}
            except Exception as e:  # keep the main line even if a variant fails
                out["variants"] = {"error": repr(e)}
        if not args.no_variants:
            try:
                out["next_rows"] = run_next_rows(torch, L, wl, K, hbm_peak)
            except Exception as e:  # keep the main line even if a row fails
                out["next_rows"] = {"error": repr(e)}
        if not args.no_cpu_baseline:
            out["cpu_baseline"] = cpu_baseline(scene_np, cam, gt_np)
        print(json.dumps(out), flush=True)
    if world > 1:
        dist.destroy_process_group()


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.impl == "reference":
        run_reference(args, rank)
        return
    run_ours(args, rank, world, local)


if __name__ == "__main__":
    main()
