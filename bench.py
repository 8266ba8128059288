"""Benchmark: decays/s of the GB300 dose engine on the synthetic adult PET/CT
phantom (256x256x300 voxels of 2x2x3 mm, 18F, 1e9 decays per step).

One step = one nm_dose_run(1e9 decays) through the C ABI: source sampling,
Woodcock transport, tally and the fold of its 10 batches (every row of the
hot path), on inputs already resident in HBM.  ``e2e`` repeats the step end
to end from pinned host buffers: CT numbers -> phantom, create (activity and
labels uploaded, alias table built), run, and the dose-rate and sigma maps
copied back.

``--impl reference`` times the FP64 CPU oracle on the same workload (a bounded
sample of decays per step) on the host cores.
Multi-GPU (torchrun): every rank simulates its own disjoint range of history
ids on its own GPU; no collective on the data path (weak scaling).
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

SHAPE = (300, 256, 256)
SPACING = (0.2, 0.2, 0.3)
DECAYS_PER_STEP = 1_000_000_000
WORKLOAD = "adult PET/CT phantom 256x256x300 voxels of 2x2x3 mm, 18F decays (2 x 511 keV + 0.25 MeV local), 27 organs, 1e9 decays per step, 10 batches"
METRIC = "decays/s"


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class Clocks:
    """nvidia-smi samples during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def __enter__(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.f.close()

    def summary(self):
        if not self.path or not os.path.exists(self.path):
            return None
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            t = [x.strip() for x in line.split(",")]
            if len(t) < 9:
                continue
            try:
                sm.append(float(t[1]))
                mx.append(float(t[2]))
            except ValueError:
                continue
            for n, v in zip(names, t[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def _phantom():
    from paper_2111_11687_gb300 import inputs
    return inputs.adult_phantom(shape=SHAPE, spacing=SPACING, seed=1)


def _materials_gpu(nm):
    from paper_2111_11687_gb300 import inputs
    return nm.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)


def _peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        return None


def _batch_phantom(i):
    from paper_2111_11687_gb300 import inputs
    ph = inputs.batch_phantoms(1, seed0=1 + i)[0]
    return ph.hu, ph.activity, ph.labels, ph.spacing


def batch_phantoms(n):
    """The batched-patients workload, generated in a spawn pool before any GPU work."""
    import multiprocessing as mp
    with mp.get_context("spawn").Pool(min(n, os.cpu_count() or 1)) as pool:
        return pool.map(_batch_phantom, range(n))


def batched_perf(torch, nm, phs, decays, steps, warmup):
    """nm_dose_run_batch over the uneven patients: every patient gets `decays`
    decays per step, the patients' launches side by side on four streams."""
    from paper_2111_11687_gb300 import inputs
    gm = _materials_gpu(nm)
    hs = []
    for hu, act, lab, sp in phs:
        den = torch.empty(hu.shape, dtype=torch.float32, device="cuda")
        mat = torch.empty(hu.shape, dtype=torch.uint8, device="cuda")
        nm.nm_ct_to_phantom(torch.from_numpy(hu).cuda(), den, mat)
        hs.append(nm.Dose(den, mat, sp, gm, activity=torch.from_numpy(act).cuda(), labels=torch.from_numpy(lab).cuda(),
                          n_labels=inputs.N_LABELS, activity_bq=inputs.ACTIVITY_BQ))
    for _ in range(warmup):
        nm.nm_dose_run_batch(hs, [decays] * len(hs), 1)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(steps):
        nm.nm_dose_run_batch(hs, [decays] * len(hs), 1)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    vox = [int(np.prod(p[0].shape)) for p in phs]
    c = hs[0].counters()
    out = {"patients": len(hs), "decays_per_patient_per_step": decays, "steps": steps,
           "value": decays * len(hs) * steps / dt, "unit": METRIC, "ms_per_step": 1e3 * dt / steps,
           "voxels_min_max": [min(vox), max(vox)],
           "launch_shape": {k: c[k] for k in ("block_threads", "chunk", "regroup", "regroup_lanes")}}
    for h in hs:
        h.close()
    return out


def run_gpu(args):
    phs = batch_phantoms(args.batch_patients) if args.batch_patients > 0 else None
    import torch

    from paper_2111_11687_gb300 import build, inputs, nmdose

    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    build.build()
    nmdose.load()
    probes = measure_ceilings(nmdose)
    ph = _phantom()
    V = ph.hu.size
    stream = torch.cuda.current_stream()
    hu_d = torch.from_numpy(ph.hu).cuda()
    den_d = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    mat_d = torch.empty(SHAPE, dtype=torch.uint8, device="cuda")
    nmdose.nm_ct_to_phantom(hu_d, den_d, mat_d, stream=stream)
    act_d = torch.from_numpy(ph.activity).cuda()
    lab_d = torch.from_numpy(ph.labels).cuda()
    gm = _materials_gpu(nmdose)
    opts = dict(n_labels=inputs.N_LABELS, activity_bq=inputs.ACTIVITY_BQ, stream=stream)
    d = nmdose.Dose(den_d, mat_d, SPACING, gm, activity=act_d, labels=lab_d, **opts)

    def barrier():
        torch.cuda.synchronize()
        if ws > 1:
            import torch.distributed as dist
            dist.barrier()
            torch.cuda.synchronize()

    seed = 1
    # Ranks take disjoint contiguous history-id ranges (no exchange while they
    # run); each rank's warm-up and timed steps continue through its range.
    from paper_2111_11687_gb300 import shard
    first, _ = shard.history_range(ws * (args.warmup + args.steps) * DECAYS_PER_STEP, ws, rank)
    d.seek(first)
    for _ in range(args.warmup):
        d.run(DECAYS_PER_STEP, seed=seed)
    c0 = d.counters()
    barrier()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with Clocks(local) as clk:
        ev0.record(stream)
        for _ in range(args.steps):
            d.run(DECAYS_PER_STEP, seed=seed)
        ev1.record(stream)
        barrier()
    ms = ev0.elapsed_time(ev1)
    c1 = d.counters()
    clocks = clk.summary()
    t_ms = torch.tensor([ms], dtype=torch.float64)
    if ws > 1:
        import torch.distributed as dist
        t_ms = t_ms.cuda()
        dist.all_reduce(t_ms, op=dist.ReduceOp.MAX)
        t_ms = t_ms.cpu()
    ms = float(t_ms.item())
    decays = DECAYS_PER_STEP * args.steps * ws
    value = decays / (ms * 1e-3)
    steps_dec = DECAYS_PER_STEP * args.steps
    transport_ms = c1["transport_ms"] - c0["transport_ms"]
    # a step's batches share one transport launch
    launch_ms = transport_ms / args.steps
    dsteps = c1["steps"] - c0["steps"]
    deps = (c1["compton"] - c0["compton"]) + (c1["photo"] - c0["photo"]) + (c1["cutoff"] - c0["cutoff"])
    per_decay = {"flight_steps": dsteps / steps_dec,
                 "interactions": (c1["compton"] - c0["compton"] + c1["photo"] - c0["photo"]) / steps_dec,
                 "positron_deposits": 1.0 if c1["emitted"] - c0["emitted"] > 2 * steps_dec * round(0.511 * 64e6) else 0.0,
                 "escapes": (c1["escapes"] - c0["escapes"]) / steps_dec}
    roofline = transport_roofline(per_decay, DECAYS_PER_STEP, launch_ms, clocks, probes)
    dose_map = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    nmdose.nm_dose_get(d.h, dose_map, None, None)
    d.close()
    variants = (variant_perf(nmdose, (den_d, mat_d, act_d, lab_d), gm, opts, args.variant_decays)
                if args.variant_decays > 0 and rank == 0 else None)

    # ---- end to end through the C ABI from pinned host buffers ---------------
    e2e = None
    if args.e2e_steps > 0:
        pin = lambda a: torch.from_numpy(a).pin_memory()
        hu_h, act_h, lab_h = pin(ph.hu), pin(ph.activity), pin(ph.labels)
        dose_h = torch.empty(SHAPE, dtype=torch.float32).pin_memory()
        sig_h = torch.empty(SHAPE, dtype=torch.float32).pin_memory()
        organ = np.zeros(inputs.N_LABELS + 1)

        def e2e_step(s):
            den2 = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
            mat2 = torch.empty(SHAPE, dtype=torch.uint8, device="cuda")
            nmdose.nm_ct_to_phantom(hu_h, den2, mat2, stream=stream)
            h = nmdose.nm_dose_create(den2, mat2, SPACING, gm, act_h, lab_h, nmdose.options(**opts))
            try:
                nmdose.nm_dose_run(h, DECAYS_PER_STEP, s)
                nmdose.nm_dose_get(h, dose_h, sig_h, organ)
            finally:
                nmdose.nm_dose_destroy(h)

        e2e_step(2)
        barrier()
        t0 = time.perf_counter()
        for _ in range(args.e2e_steps):
            e2e_step(3)
        barrier()
        e2e_s = time.perf_counter() - t0
        e2e_val = DECAYS_PER_STEP * args.e2e_steps * ws / e2e_s
        e2e = {"value": e2e_val, "unit": METRIC, "h2d_bytes_per_step": int(V * (2 + 4 + 1)),
               "d2h_bytes_per_step": int(V * 8 + 8 * (inputs.N_LABELS + 1)), "steps": args.e2e_steps}

    den = (denoiser_perf(torch, nmdose, args.denoiser_steps, _peaks(), (dose_map, den_d, act_d))
           if args.denoiser_steps > 0 else None)
    batched = batched_perf(torch, nmdose, phs, args.batch_decays, 3, 1) if phs else None

    ttt = time_to_2pct(args) if rank == 0 and ws == 1 and args.ttt_train > 0 else None
    if ttt is not None and args.whole_body:
        ttt["whole_body"] = whole_body_time_to_2pct()
    cpu = None
    if rank == 0 and ws == 1 and args.cpu_decays > 0:
        cpu = cpu_baseline(args.cpu_decays)
    if rank == 0:
        # transport + fold + organ fold per step
        launches = 3 * args.steps
        line = {"metric": METRIC, "value": value, "unit": METRIC, "n_gpus": ws, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f32+int64", "data": "synthetic",
                "config": {"workload": WORKLOAD, "decays_per_step": DECAYS_PER_STEP, "grid": list(SHAPE[::-1]),
                           "voxel_mm": [x * 10 for x in SPACING], "batches": 10,
                           "l2": "working set (tallies 11x157 MB + grid 79 MB + alias 41 MB) exceeds the 129 MB L2",
                           "parallelism": f"histories sharded over {ws} GPU(s)"},
                "gpu_launches": launches, "roofline": roofline, "clocks": clocks, "e2e": e2e,
                "cpu_baseline": cpu, "denoiser": den, "batched": batched, "time_to_2pct": ttt,
                "variants": variants}
        print(json.dumps(line))
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def variant_perf(nm, arrays, gm, opts, decays):
    """Decays/s of the transport variants on the benchmark phantom (device
    time of the transport launches): 18F with history-by-history sigma (and
    the fraction of histories whose deposits spread over more voxels than a
    lane keeps), 18F with the beta+ spectrum and positron tracks, 177Lu and
    131I (beta- tracks, gamma lines, no annihilation pair)."""
    from paper_2111_11687_gb300 import nuclides
    den, mat, act, lab = arrays
    cases = {"18F_history_sigma": dict(history_sigma=1), "18F_beta_tracks": nuclides.F18_TRACKED,
             "177Lu": nuclides.LU177, "131I": nuclides.I131}
    out = {}
    for name, kw in cases.items():
        with nm.Dose(den, mat, SPACING, gm, activity=act, labels=lab, **opts, **kw) as d:
            d.run(decays // 5, seed=1)
            c0 = d.counters()
            d.run(decays, seed=2)
            c1 = d.counters()
        ms = c1["transport_ms"] - c0["transport_ms"]
        r = {"decays_per_s": decays / (ms * 1e-3), "emitted_mev_per_decay":
             (c1["emitted"] - c0["emitted"]) / 64e6 / decays}
        if name == "18F_history_sigma":
            r["split_histories_fraction"] = (c1["history_splits"] - c0["history_splits"]) / decays
        out[name] = r
    return out


def time_to_2pct(args):
    """The second half of the metric: wall time until every one of the 27
    organ doses is within 2 % of a 1e10-decay plain-MC reference, plain MC
    against MC + denoiser, on held-out adult phantoms (256x256x300 x 2x2x3 mm).

    The denoiser is trained in this run by the library's own kernels, on
    pairs the engine generates (1e7 -> 1e9 decays) on ``--ttt-train`` seeded
    phantoms; ``--ttt-candidates`` networks train and the one with the lowest
    loss on a held-out tenth of the training phantoms is kept.  Plain MC
    checks the organ means every 5e6 decays; MC + denoiser denoises the
    accumulated map every 1e7 decays (inference on the organs' bounding box)
    and stops at the first checkpoint that passes.  Both arms are timed on
    the host around device-synchronised work, per phantom."""
    from paper_2111_11687_gb300 import experiment
    t0 = time.perf_counter()
    r = experiment.run(train_n=args.ttt_train, test_n=args.ttt_test, steps=args.ttt_steps,
                       candidates=args.ttt_candidates)
    cases = [{"plain_mc_ms": None if c["plain_mc_s"] is None else 1e3 * c["plain_mc_s"],
              "plain_mc_decays": c["plain_mc_decays"],
              "mc_denoiser_ms": None if c["mc_denoiser_s"] is None else 1e3 * c["mc_denoiser_s"],
              "mc_denoiser_decays": c["mc_denoiser_decays"],
              "denoiser_wins": c["mc_denoiser_s"] is not None and
              (c["plain_mc_s"] is None or c["mc_denoiser_s"] < c["plain_mc_s"]),
              "worst_organ_err_1e7_raw": c["low_mc_max_err"], "worst_organ_err_1e7_denoised": c["denoiser_max_err"]}
             for c in r["cases"]]
    return {"workload": "held-out adult phantoms 256x256x300 x 2x2x3 mm, 27 organs, target <= 2 % on every organ "
                        "against a 1e10-decay plain-MC reference",
            "test_phantoms": r["test"], "reference_decays": r["ref"],
            "plain_mc_ms_median": 1e3 * r["plain_mc_s_median"], "mc_denoiser_ms_median": 1e3 * r["mc_denoiser_s_median"],
            "plain_mc_decays_median": r["plain_mc_decays_median"],
            "mc_denoiser_decays_median": r["mc_denoiser_decays_median"],
            "denoiser_faster": r["denoiser_faster"],
            "denoiser_reaches_2pct_first_checkpoint": r["denoiser_reaches_2pct_first_checkpoint"],
            "worst_organ_err_1e7_median": {"raw": r["low_mc_max_err_median"], "denoised": r["denoiser_max_err_median"]},
            "network": {"provenance": "trained in this run", "train_phantoms": r["train"], "pairs": [r["low"], r["high"]],
                        "steps": r["steps"], "patch": r["patch"], "batch": r["batch"], "candidates": r["candidates"],
                        "final_loss": r["final_loss"], "candidate_val_losses": r["candidate_val_losses"],
                        "data_s": r["data_s"], "train_s": r["train_s"]},
            "wall_s": time.perf_counter() - t0, "per_phantom": cases}


def whole_body_time_to_2pct():
    """The whole-body workload (512x512x600 voxels of 1x1x3 mm with 1-3 cm
    lesions): plain MC's wall time until all 27 organ means are within 2 % of
    a 1e10-decay reference (organ means from the fold's sums every 5e6
    decays), and the MC + denoiser arm's cost before any check (MC of 1e8
    decays and one inference on the organs' bounding box), a lower bound of
    that arm: no network is trained at 1 x 1 x 3 mm."""
    from paper_2111_11687_gb300 import experiment
    wb = experiment.configs()["whole_body"]
    return {"grid": wb["grid"], "voxel_mm": wb["voxel_mm"], "reference_decays": wb["reference_decays"],
            "plain_mc_ms": None if wb["plain_mc_s"] is None else 1e3 * wb["plain_mc_s"],
            "plain_mc_decays": wb["plain_mc_decays"], "plain_mc_worst_organ_err": wb["plain_mc_err"],
            "mc_denoiser_lower_bound_ms": 1e3 * wb["mc_denoiser_lower_bound_s"],
            "decays_per_s_1e9": wb["decays_per_s_1e9"]}


def measure_ceilings(nm):
    """This GPU's L2 read bandwidth (48 MiB buffer, far below the 129 MB L2)
    and scattered 64-bit atomic-add rate (16 MiB of slots), measured by the
    library's probes with CUDA events; both are ceilings of the transport."""
    return {"l2_read_gbs": nm.nm_probe_l2_read(48 << 20, 40),
            "atomic_add_u64_per_s": nm.nm_probe_atomic_add_u64(1 << 21, 1 << 28)}


def _profile_figures():
    """Figures of the committed ncu summary of the transport kernel, used only
    while the kernel source is the one that was profiled (keyed by hash)."""
    tp = os.path.join(ROOT, "profiles", "transport_kernel_adult_phantom.md")
    if not os.path.exists(tp):
        return None
    kv = {}
    for line in open(tp):
        if ":" in line and not line.startswith(("|", " ", "#")):
            k, v = line.split(":", 1)
            kv[k.strip()] = v.strip()
    if kv.get("kernel_source_hash") != _kernel_hash():
        return None
    out = {}
    for k in ("dram_bytes_per_decay", "lts_sectors_per_decay", "issue_active_pct", "lane_efficiency_pct",
              "warp_inst_per_decay", "dram_busy_pct"):
        if k in kv:
            out[k] = float(kv[k])
    return out


def transport_roofline(per_decay, decays_per_launch, launch_ms, clocks, probes, sms=152, schedulers=4):
    """Roofline of the transport kernel.

    Memory view (the headline ``frac``): algorithmic bytes per decay = 5 B per
    voxel read (FP32 density + u8 material, one per flight step) + 8 B per
    int64 tally atomic (one per interaction and per positron deposit) + 12 B
    per alias entry (one per decay), times the decays of one launch, over the
    launch's average CUDA-event time, against the measured HBM copy peak.
    Further ceilings: the measured L2 read bandwidth (sector view, from the
    profile's L2 sectors per decay), the measured scattered atomic rate, and
    instruction issue (the profile's warp instructions per decay against SMs x
    schedulers x the sampled SM clock)."""
    peaks = _peaks()
    hbm = peaks["hbm_gbs"] if peaks else 6800.0
    atomics = per_decay["interactions"] + per_decay["positron_deposits"]
    bytes_per_decay = 5.0 * per_decay["flight_steps"] + 8.0 * atomics + 12.0
    decays_per_s = decays_per_launch / (launch_ms * 1e-3)
    achieved = bytes_per_decay * decays_per_s / 1e9
    prof = _profile_figures()
    traffic = prof["dram_bytes_per_decay"] * decays_per_launch if prof and "dram_bytes_per_decay" in prof else None
    ceilings = {}
    if probes:
        if prof and "lts_sectors_per_decay" in prof:
            l2 = prof["lts_sectors_per_decay"] * 32.0 * decays_per_s / 1e9
            ceilings["l2_sectors"] = {"achieved": l2, "peak": probes["l2_read_gbs"], "unit": "GB/s",
                                      "frac": l2 / probes["l2_read_gbs"], "source": "ncu L2 sectors per decay x 32 B"}
        rate = atomics * decays_per_s
        ceilings["atomics"] = {"achieved": rate, "peak": probes["atomic_add_u64_per_s"], "unit": "atomics/s",
                               "frac": rate / probes["atomic_add_u64_per_s"], "per_decay": atomics}
    if prof and "warp_inst_per_decay" in prof and clocks and clocks.get("sm_mhz"):
        cap = sms * schedulers * clocks["sm_mhz"] * 1e6 / prof["warp_inst_per_decay"]
        ceilings["issue"] = {"achieved": decays_per_s, "peak": cap, "unit": "decays/s", "frac": decays_per_s / cap,
                             "warp_inst_per_decay": prof["warp_inst_per_decay"],
                             "lane_efficiency_pct": prof.get("lane_efficiency_pct")}
    return {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": achieved / hbm,
            "traffic": traffic,
            "traffic_source": "from_profile: profiles/transport_kernel_adult_phantom.md (same kernel source)"
            if traffic is not None else None,
            "peak_source": "measured" if peaks else "fallback", "kernel": "transport_ring_kernel",
            "launch_ms": launch_ms, "decays_per_launch": decays_per_launch, "bytes_per_decay": bytes_per_decay,
            "per_decay": per_decay, "ceilings": ceilings, "probes": probes}


def unet_flops(layers, patch, batch, levels=4):
    """Dense FLOPs of the U-Net's 3x3x3 convolutions for one batch (2 per MAC,
    the 27*cin real K, not the padded one)."""
    f = 0
    names = []
    for i in range(levels):
        names += [i, i]
    for i in range(levels - 2, -1, -1):
        names += [i, i]
    for l, lev in zip(layers[:-1], names):
        vox = batch * (patch >> lev) ** 3
        f += 2 * vox * l["cout"] * 27 * l["cin"]
    return f


def infer_box(density, margin=8, align=8):
    """Voxels of the volume that whole-volume inference runs: the body's
    bounding box (density >= 0.1) plus the context margin, each side rounded
    up to the network's alignment."""
    idx = (density >= 0.1).nonzero()
    ext = (idx.max(0).values - idx.min(0).values + 1 + 2 * margin).tolist()
    return [(e + align - 1) // align * align for e in ext]


def denoiser_perf(torch, nm, steps, peaks, vol=None):
    """Forward and training-step throughput of the U-Net (64^3 patches, batch 4)
    on the tensor cores, timed with CUDA events on the launching stream; with
    vol = (dose, density, activity), also whole-volume inference on it."""
    P, B = 64, 4
    stream = torch.cuda.current_stream()
    net = nm.Denoiser(patch=P, batch=B, levels=4, base_width=16, seed=1, stream=stream)
    rng = np.random.default_rng(0)
    x = torch.from_numpy(rng.normal(0, 1, (B, P, P, P, 8)).astype(np.float32)).to(torch.bfloat16).cuda()
    t = torch.from_numpy(rng.normal(0, 1, (B, P, P, P)).astype(np.float32)).cuda()
    y = torch.empty((B, P, P, P), dtype=torch.float32, device="cuda")
    fl = unet_flops(net.layers(), P, B)
    for _ in range(3):
        net.forward(x, y)
        net.train_step(x, t, lr=1e-4)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    torch.cuda.synchronize()
    e[0].record(stream)
    for _ in range(steps):
        net.forward(x, y)
    e[1].record(stream)
    for _ in range(steps):
        net.train_step(x, t, lr=1e-4)
    e[2].record(stream)
    torch.cuda.synchronize()
    fwd_ms = e[0].elapsed_time(e[1]) / steps
    trn_ms = e[1].elapsed_time(e[2]) / steps
    peak = peaks["bf16_tflops"] if peaks else 1900.0
    fwd_tf = fl / (fwd_ms * 1e-3) / 1e12
    trn_tf = 3 * fl / (trn_ms * 1e-3) / 1e12      # forward + input and weight gradients
    out = {"patch": P, "batch": B, "widths": [16, 32, 64, 128], "forward_ms": fwd_ms, "train_step_ms": trn_ms,
           "forward_gflop": fl / 1e9, "patches_per_s_forward": B / (fwd_ms * 1e-3),
           "roofline": {"bound": "tensor", "achieved": fwd_tf, "peak": peak, "unit": "TFLOP/s",
                        "frac": fwd_tf / peak, "train_achieved": trn_tf, "train_frac": trn_tf / peak,
                        "peak_source": "measured" if peaks else "fallback"}}
    if vol is not None:
        dose, density, act = vol
        res = torch.empty_like(dose)
        net.apply(dose, density, act, res)   # allocates the inference buffers
        torch.cuda.synchronize()
        e[0].record(stream)
        for _ in range(steps):
            net.apply(dose, density, act, res)
        e[1].record(stream)
        torch.cuda.synchronize()
        ap_ms = e[0].elapsed_time(e[1]) / steps
        box = infer_box(density)
        fl_box = unet_flops(net.layers(), P, 1) * (box[0] * box[1] * box[2]) / P ** 3
        ap_tf = fl_box / (ap_ms * 1e-3) / 1e12
        out["apply"] = {"volume": list(dose.shape[::-1]), "network_box_zyx": box, "ms": ap_ms, "tflops": ap_tf,
                        "frac": ap_tf / peak}
    net.close()
    return out


def _kernel_hash():
    import hashlib
    h = hashlib.sha256()
    for f in ("nm_transport.cu", "nm_internal.cuh"):
        h.update(open(os.path.join(ROOT, "paper_2111_11687_gb300", "csrc", f), "rb").read())
    return h.hexdigest()[:16]


def cpu_baseline(n_decays):
    """The FP64 oracle on the same phantom, on all host cores, bounded sample."""
    import oracle
    from paper_2111_11687_gb300 import inputs
    oracle.build()
    ph = _phantom()
    den, mat = oracle.hu_to_phantom(ph.hu)
    om = oracle.Materials(inputs.MATERIAL_Z_OVER_A, inputs.MATERIAL_ZEFF, inputs.PE_COEFF, inputs.PE_EXP)
    t0 = time.perf_counter()
    r = oracle.run(den, mat, om, activity=ph.activity, labels=ph.labels, n_labels=inputs.N_LABELS,
                   spacing=SPACING, n_hist=n_decays, seed=1, batches=10, activity_bq=inputs.ACTIVITY_BQ)
    dt = time.perf_counter() - t0
    return {"value": n_decays / dt, "unit": METRIC, "cores": r.counters["threads_used"], "kind": "oracle",
            "sample": f"{n_decays} decays of the same phantom (FP64, Siddon traversal), {dt:.1f} s"}


def run_reference(args):
    ws, rank, _ = _dist()
    if rank != 0:
        return
    n = args.ref_decays
    for _ in range(args.warmup):
        pass  # the oracle has no warm-up state; each step is a fresh bounded sample
    vals = []
    t_total = 0.0
    for _ in range(args.steps):
        c = cpu_baseline(n)
        vals.append(c["value"])
        t_total += n / c["value"]
    value = n * args.steps / t_total
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": METRIC, "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_total / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": WORKLOAD, "decays_per_step": n},
            "cpu_baseline": {"value": value, "unit": METRIC, "cores": c["cores"], "kind": "oracle",
                             "sample": f"{args.steps} x {n} decays of the benchmark phantom"},
            "e2e": {"value": value, "unit": METRIC, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


def run_profile(args):
    """One short run of the benchmark workload for ncu: create, then one
    nm_dose_run of --decays decays in 2 batches (one transport launch)."""
    import torch

    from paper_2111_11687_gb300 import build, inputs, nmdose
    build.build()
    ph = _phantom()
    den = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    mat = torch.empty(SHAPE, dtype=torch.uint8, device="cuda")
    nmdose.nm_ct_to_phantom(torch.from_numpy(ph.hu).cuda(), den, mat)
    with nmdose.Dose(den, mat, SPACING, _materials_gpu(nmdose), activity=torch.from_numpy(ph.activity).cuda(),
                     labels=torch.from_numpy(ph.labels).cuda(), n_labels=inputs.N_LABELS, batches=2,
                     activity_bq=inputs.ACTIVITY_BQ, **json.loads(args.tuning)) as d:
        d.run(args.decays, seed=1)
        c = d.counters()
    torch.cuda.synchronize()
    print(json.dumps({"profile_decays": args.decays, "transport_ms": c["transport_ms"],
                      "decays_per_s": args.decays / (c["transport_ms"] * 1e-3), "counters": c}))


def run_apply(args):
    """Whole-volume denoiser inference on the benchmark phantom, for ncu: a
    dose map of --decays decays, then --apply-reps applies of a fresh network
    (the time does not depend on the weights)."""
    import torch

    from paper_2111_11687_gb300 import build, inputs, nmdose
    build.build()
    ph = _phantom()
    den = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    mat = torch.empty(SHAPE, dtype=torch.uint8, device="cuda")
    nmdose.nm_ct_to_phantom(torch.from_numpy(ph.hu).cuda(), den, mat)
    act = torch.from_numpy(ph.activity).cuda()
    dose = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    with nmdose.Dose(den, mat, SPACING, _materials_gpu(nmdose), activity=act, labels=torch.from_numpy(ph.labels).cuda(),
                     n_labels=inputs.N_LABELS, activity_bq=inputs.ACTIVITY_BQ, **json.loads(args.tuning)) as d:
        d.run(args.decays, seed=1)
        nmdose.nm_dose_get(d.h, dose, None, None)
    net = nmdose.Denoiser(patch=64, batch=4, levels=4, base_width=16, seed=1)
    out = torch.empty_like(dose)
    t = []
    for _ in range(args.apply_reps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        net.apply(dose, den, act, out)
        torch.cuda.synchronize()
        t.append((time.perf_counter() - t0) * 1e3)
    net.close()
    print(json.dumps({"apply_decays": args.decays, "apply_ms": t, "network_box_zyx": infer_box(den)}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--e2e-steps", type=int, default=4)
    ap.add_argument("--cpu-decays", type=int, default=12_000_000)
    ap.add_argument("--ref-decays", type=int, default=6_000_000)
    ap.add_argument("--denoiser-steps", type=int, default=10)
    ap.add_argument("--batch-patients", type=int, default=16)
    ap.add_argument("--batch-decays", type=int, default=100_000_000)
    ap.add_argument("--variant-decays", type=int, default=500_000_000,
                    help="decays per transport variant (history sigma, beta tracks, 177Lu, 131I; 0 = skip)")
    ap.add_argument("--ttt-train", type=int, default=200, help="time-to-2%% block: training phantoms (0 = skip)")
    ap.add_argument("--ttt-test", type=int, default=20, help="time-to-2%% block: held-out phantoms")
    ap.add_argument("--ttt-steps", type=int, default=10000, help="time-to-2%% block: training steps per network")
    ap.add_argument("--ttt-candidates", type=int, default=3, help="time-to-2%% block: networks trained")
    ap.add_argument("--whole-body", type=int, default=1, help="time-to-2%% block: add the whole-body phantom")
    ap.add_argument("--denoiser-only", action="store_true", help="only the U-Net throughput (for ncu)")
    ap.add_argument("--profile", action="store_true", help="one short run for ncu")
    ap.add_argument("--decays", type=int, default=200_000_000)
    ap.add_argument("--tuning", default="{}", help="JSON dict of nm_options launch fields (profile mode)")
    ap.add_argument("--apply-only", action="store_true", help="only whole-volume denoiser inference (for ncu)")
    ap.add_argument("--apply-reps", type=int, default=1)
    args = ap.parse_args()
    if args.denoiser_only:
        import torch

        from paper_2111_11687_gb300 import build, nmdose
        build.build()
        print(json.dumps(denoiser_perf(torch, nmdose, args.denoiser_steps, _peaks())))
    elif args.profile:
        run_profile(args)
    elif args.apply_only:
        run_apply(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
