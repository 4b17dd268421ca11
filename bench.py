"""Throughput bench of the GB300 SND hot path.

Workload: one full Northern Cross beam - 1024 channels over 400-416 MHz, dt = 0.138 ms,
2048 trial DMs over 0-2000 pc cm^-3, uint8 filterbank streamed in 16384-sample chunks,
seeded synthetic noise with 200 injected bursts. A step streams 16 chunks (2^18 samples)
through the whole path (encoder -> SND tree -> matched filter -> candidates) in each of the
three modes (binary, graded, float; branching 8, Supplementary Table S1 operating points);
the three plans keep streaming across steps, so every timed chunk emits 16384 samples per
DM row. Metric: DM-trial samples per second (DM rows x emitted plane samples / time).

Multi-GPU: beams are independent, so N ranks run N beam replicas with no collective
(weak scaling); value = all ranks' DM-samples / the slowest rank's time.

--impl reference runs the C++/OpenMP CPU oracle (the only other implementation of this method
here) on bounded samples of the same workload on all host cores.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import synth  # noqa: E402

W = synth.NC1024
MODES = (("binary", 0), ("graded", 1), ("float", 2))
BRANCHING = 8
TREE_BYTES_PER_DM_SAMPLE = W.nchan / W.ndm + 4.0  # uint8 input read once + int32 plane written once
# ALU-pipe ceiling of the bit-sliced tree. The logic and shift instructions that make up the
# tree's arithmetic (LOP3, SHF) issue on each SM sub-partition's ALU pipe at 16 lanes per cycle
# (ncu's pipe_alu peak of 0.5 warp-instructions per cycle), so a GPU retires
# SMs x 4 x 16 x clock of them per second. The work the direct kernel cannot avoid, in those
# operations per DM-sample (a 32-sample word per operation):
#   float / graded: per channel one funnel shift (align the channel's word to the DM's delay)
#     and one carry-save full adder (two LOP3) -> 3 N_f / 32;
#   binary (C = 4): per leaf four funnel shifts, the quorum (three LOP3) and the parent's
#     thermometer (two LOP3) -> 9 N_f / (4 * 32).
ALU_LANES_PER_SM_CYCLE = 4 * 16
DATA_NOTE = "synthetic: seeded rint(N(128,16)) uint8 noise + 200 injected dispersed bursts"


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.proc = None
        self.lines = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread:
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
            for name, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def _traffic_from_profile(src_hash: str):
    """DRAM bytes per tree launch from the committed ncu summary, if it was taken on this
    exact tree kernel source (else None)."""
    path = os.path.join(ROOT, "profiles", "k_snd_nc1024_2048dm.md")
    try:
        txt = open(path).read()
    except OSError:
        return None
    vals = {}
    for line in txt.splitlines():
        if line.startswith("bench_key:"):
            k, _, v = line[len("bench_key:"):].strip().partition("=")
            vals[k.strip()] = v.strip()
    if vals.get("tree_source_sha1") != src_hash:
        return None
    try:
        return float(vals["dram_bytes_per_full_launch"])
    except (KeyError, ValueError):
        return None


def _tree_source_hash() -> str:
    import hashlib
    h = hashlib.sha1()
    for f in ("tree_direct.cu", "snd_internal.h"):
        with open(os.path.join(ROOT, "paper_2606_15361_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


def reduce_max(values, dist=None, device=None):
    """Max over ranks of per-rank timings (the slowest rank sets the whole-job time)."""
    if dist is None or not dist.is_initialized() or dist.get_world_size() == 1:
        return [float(v) for v in values]
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t.cpu()]


def whole_job_rate(units_per_rank_step: float, steps: int, world: int, ms: float) -> float:
    """Units processed by all ranks (weak scaling: each rank its own beam replica) per second
    of the slowest rank."""
    return units_per_rank_step * steps * world / (ms / 1e3)


# ----------------------------------------------------------------------------------------
# CPU oracle (reference arm and cpu_baseline)
# ----------------------------------------------------------------------------------------

def _cxx_streams(chunks, fill: int = 2):
    """One C++-oracle stream per mode, filled with the first `fill` chunks (from then on
    every chunk emits W.chunk plane samples per DM row)."""
    from oracle import cxx
    from oracle import stream as ost
    out = {}
    for name, m in MODES:
        s = cxx.Stream(W.freqs(), synth.NC_DT, W.dms(), ost.defaults(m, branching=BRANCHING))
        for i in range(fill):
            s.push(chunks[i], want_plane=False)
        out[name] = s
    return out


def oracle_sample(chunks):
    """The C++/OpenMP oracle (oracle/cpp, as it stands) timed on the host cores on bounded
    samples of the workload. Returns the cpu_baseline object:
    * value: the whole path (encoder, SND tree per DM with no sharing, matched filter,
      closing + labelling) on one steady-state chunk of the bench beam in each of the three
      modes, all cores, in DM-samples/s;
    * brute_force: direct dedispersion of one chunk (all 2048 rows), all cores;
    * single_thread: the same whole-path chunk in float mode on one core, over a bounded
      sample of rows (the tree and matched filter of 128 rows; the encoder of all channels);
    * c1_full: the 64-channel / 128-DM beam (one 16384-sample chunk, binary, B = 2) in full,
      all cores and one core."""
    from oracle import cxx
    from oracle import stream as ost
    ncpu = cxx.max_threads()
    streams = _cxx_streams(chunks)
    t0 = time.perf_counter()
    work = 0
    for name, _ in MODES:
        r = streams[name].push(chunks[2], want_plane=False)
        work += W.ndm * (r["e_new"] - r["e_prev"])
    secs = time.perf_counter() - t0
    out = {"value": work / secs, "unit": "DM-samples/s", "cores": ncpu, "kind": "oracle",
           "sample": "C++/OpenMP oracle, whole path (encoder, SND tree per DM without sharing, matched filter, "
                     "closing + labelling) on one steady-state 16384-sample chunk of the bench beam in each of "
                     "the three modes (B = 8), all host cores"}
    x = np.concatenate([cxx.encode_chunk(chunks[i], 1.5)[0] for i in range(3)], axis=1)
    tab = cxx.delay_table(W.freqs(), synth.NC_DT, W.dms())
    D = int(tab.max())
    t0 = time.perf_counter()
    cxx.brute_rows(x, 0, tab, range(W.ndm), 2 * W.chunk - D, W.chunk)
    secs = time.perf_counter() - t0
    out["brute_force"] = {"value": W.ndm * W.chunk / secs, "unit": "DM-samples/s", "cores": ncpu,
                          "sample": "direct dedispersion y_d(t) = sum_c x_c(t + delta_c(d)) of one chunk, 2048 rows"}
    rows = 128
    cfg = ost.defaults(2, branching=BRANCHING)
    widths = [cxx.row_widths(W.freqs(), synth.NC_DT, d, cfg.mf_alpha) for d in W.dms()[:rows]]
    cxx.set_threads(1)
    try:
        t0 = time.perf_counter()
        xe = np.concatenate([cxx.encode_chunk(chunks[i], cfg.enc_theta)[0] for i in range(3)], axis=1)
        y = cxx.snd_rows(xe, 0, tab, range(rows), 2 * W.chunk - D, W.chunk, 2, cfg.cluster, cfg.branching)
        for r in range(rows):
            cxx.row_mf(y[r], W.chunk - 1023, widths[r], cfg.det_theta)
        secs = time.perf_counter() - t0
        out["single_thread"] = {"value": rows * W.chunk / secs, "unit": "DM-samples/s", "cores": 1,
                                "sample": "float mode, one chunk: encoder (3 chunks, all channels), tree + matched "
                                          f"filter of {rows} of 2048 rows"}
        c1 = {}
        w = synth.NC64
        d64 = w.chunk_data(0)
        for label, th in (("one_core", 1), ("all_cores", ncpu)):
            cxx.set_threads(th)
            t0 = time.perf_counter()
            s = cxx.Stream(w.freqs(), synth.NC_DT, w.dms(), ost.defaults(0, branching=2))
            r = s.push(d64, want_plane=False)
            secs = time.perf_counter() - t0
            c1[label] = w.ndm * (r["e_new"] - r["e_prev"]) / secs
        out["c1_full"] = {"value": c1["all_cores"], "single_thread_value": c1["one_core"], "unit": "DM-samples/s",
                          "cores": ncpu, "sample": "64 ch, 128 DMs 0-100, one 16384-sample chunk, binary, B = 2"}
    finally:
        cxx.set_threads(ncpu)
    return out


def oracle_rows_sample(chunks):
    """The oracle timed on bounded samples of the other rows (single-threaded numpy):
    multi-rate (the NC64 beam, all bands, graded), the labelled-payload tree (FP16 storage,
    2 DM rows of the bench beam over one chunk) and the sifter's forward pass (4 snippets).
    Units are each row's own: native DM-samples/s, DM-samples/s, snippets/s."""
    from oracle import multirate as omr
    from oracle import sifter as osf
    from oracle import stream as ost
    from oracle import zpayload as oz
    out = {}
    w = synth.NC64
    t0 = time.perf_counter()
    m = omr.MultiRateStream(w.freqs(), synth.NC_DT, w.dms(), ost.defaults(ost.GRADED, branching=2))
    m.push(w.chunk_data(0))
    m.candidates()
    dt = time.perf_counter() - t0
    out["multirate"] = {"value": w.ndm * w.chunk / dt, "unit": "native DM-samples/s", "cores": 1,
                        "sample": "NC64 beam (64 ch, 128 DMs, 16384 samples), graded, bands 1/2/4/8, merge"}
    t0 = time.perf_counter()
    z = oz.ZStream(W.freqs(), synth.NC_DT, W.dms(), 4, BRANCHING, 1.5, np.float16, rows=[0, 1024])
    for c in chunks[:3]:
        z.push(c)
    dt = time.perf_counter() - t0
    emitted = z.E
    out["zfloat_fp16"] = {"value": 2 * emitted / dt, "unit": "DM-samples/s", "cores": 1,
                          "sample": "labelled payload, FP16 storage, 2 of 2048 DM rows over 3 chunks of the bench beam"}
    rng = np.random.default_rng(1)
    theta = osf.init_params(1)
    x = rng.normal(size=(4, 64, 256))
    t0 = time.perf_counter()
    osf.forward(theta, x)
    dt = time.perf_counter() - t0
    out["sifter_forward"] = {"value": 4 / dt, "unit": "snippets/s", "cores": 1, "sample": "FP64 forward of 4 snippets"}
    return out


def run_reference(args, rank, world):
    """The oracle as it stands (C++/OpenMP, all host cores) on the bench's workload: one
    step = the next steady-state 16384-sample chunk of one mode's stream, the modes in turn
    (binary, graded, float), so a step is a bounded sample of the GPU arm's step."""
    out = {"impl": "reference", "metric": "DM-trial samples/s", "unit": "DM-samples/s",
           "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "int32/f64", "data": DATA_NOTE}
    if rank != 0:
        return None
    from oracle import cxx
    total = args.warmup + args.steps
    per_mode = (total + len(MODES) - 1) // len(MODES)
    chunks = [W.chunk_data(i) for i in range(min(W.nchunks, 2 + per_mode))]
    streams = _cxx_streams(chunks)
    nxt = {name: 2 for name, _ in MODES}
    work = 0
    secs = 0.0
    for k in range(total):
        name = MODES[k % len(MODES)][0]
        i = nxt[name]
        nxt[name] = 2 + (i - 1) % (len(chunks) - 2)
        t0 = time.perf_counter()
        r = streams[name].push(chunks[i], want_plane=False)
        dt = time.perf_counter() - t0
        if k >= args.warmup:
            work += W.ndm * (r["e_new"] - r["e_prev"])
            secs += dt
    v = work / secs
    ncpu = cxx.max_threads()
    desc = ("C++/OpenMP oracle, whole path (encoder, SND tree per DM without sharing, matched filter, closing + "
            "labelling); a step = one steady-state 16384-sample chunk of one mode, modes in turn; all host cores")
    out.update({"value": v, "ms_per_step": 1e3 * secs / max(args.steps, 1),
                "config": {"workload": "nc1024_2048dm: 1024 ch 400-416 MHz, dt 0.138 ms, 2048 DMs 0-2000, "
                                       "16384-sample chunks, B=8, binary+graded+float",
                           "sample": desc},
                "cpu_baseline": {"value": v, "unit": "DM-samples/s", "cores": ncpu, "kind": "oracle", "sample": desc},
                "e2e": {"value": v, "unit": "DM-samples/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}})
    return out


# ----------------------------------------------------------------------------------------
# GPU arm
# ----------------------------------------------------------------------------------------

def multirate_rate(g, args, dev, stream, dchunks, freqs, dms, mode=("graded", 1), s_max=16):
    """Multi-rate search of the same beam (graded mode, bands up to S = 16 as in Table S1;
    each chunk's scrunching and band stages replayed as one CUDA graph), timed beside the
    single-rate plan of the same mode: native DM-samples per second."""
    import torch
    m = g.MultiRatePlan(freqs, synth.NC_DT, dms, BRANCHING, mode[1], g.options(mode[1], max_chunk=W.chunk),
                        s_max=s_max, device=dev)
    m.set_graph(True)
    single = g.Plan(freqs, synth.NC_DT, dms, BRANCHING, mode[1], g.options(mode[1], max_chunk=W.chunk), device=dev)
    steps = max(1, min(args.steps, 5))
    out = {"mode": mode[0], "s_max": s_max, "bands": [[s, n] for s, n in zip(m.scrunch, m.band_ndm)]}
    for name, run in (("multirate", lambda c: m.execute(c)), ("single_rate", lambda c: single.execute(c))):
        for _ in range(max(args.warmup, 1)):
            for c in dchunks:
                run(c)
        (m if name == "multirate" else single).candidates(check=False)
        torch.cuda.synchronize(dev)
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        for _ in range(steps):
            for c in dchunks:
                run(c)
        ev1.record(stream)
        torch.cuda.synchronize(dev)
        ms = ev0.elapsed_time(ev1) / steps
        out[name] = {"ms_per_step": ms, "dm_samples_per_s": W.nchunks * W.chunk * W.ndm / (ms / 1e3)}
    t0 = time.perf_counter()
    c, _ = m.candidates(check=False)
    out["merge_ms"] = 1e3 * (time.perf_counter() - t0)
    out["merged_candidates"] = int(len(c))
    out["speedup"] = out["single_rate"]["ms_per_step"] / out["multirate"]["ms_per_step"]
    out["note"] = "step = 16 chunks of 16384 native samples; merge (candidate read) timed once, host clock"
    return out


def branching_sweep(g, args, dev, dchunks, freqs, dms, branchings=(2, 4, 8)):
    """Tree time per steady 16384-sample chunk of the bench beam for each branching factor and
    mode (the factor is free in Methods, "Tree levels"; float and uncapped graded planes do
    not depend on it), from the stage events, with the HBM fraction on 4.5 B per DM-sample."""
    peaks, src = _peaks()
    out = {}
    for B in branchings:
        row = {}
        for name, m in MODES:
            p = g.Plan(freqs, synth.NC_DT, dms, B, m, g.options(m, max_chunk=W.chunk), device=dev)
            for c in dchunks[:3]:
                p.execute(c)
            p.profile(True)
            p.profile_read()
            for c in dchunks[3:8]:
                p.execute(c)
            prof = p.profile_read()
            tms = prof["tree"][0] / max(prof["tree"][1], 1)
            ach = TREE_BYTES_PER_DM_SAMPLE * W.chunk * W.ndm / (tms / 1e3) / 1e9
            row[name] = {"tree_ms_per_chunk": round(tms, 4), "hbm_frac": round(ach / peaks["hbm_gbs"], 4),
                         "kernel": g.TREE_KERNELS[p.stats().tree_kernel], "levels": int(p.stats().nlevels)}
            del p
        out[str(B)] = row
    out["note"] = ("tree stage per chunk (CUDA events), 5 steady chunks after 3 warm-up; hbm_frac of the measured "
                   f"copy bandwidth ({src})")
    return out


def stress_rate(g, args, dev, nbeams=16):
    """Stress scale (4096 channels 400-416 MHz, dt 0.138 ms, 8192 DMs over 0-3000, 1 s chunks
    of 7246 samples, B = 4; graded and float): per mode, one beam's tree time per chunk and its
    HBM fraction on 4.5 B per DM-sample, and the L2-residency sweep: steps of k = 1..16 beams
    advanced together through the batch API (the bit rings of k beams, 26 MB each, are the
    working set the 129 MB L2 holds or not), in whole-step DM-samples per second."""
    import torch
    from concurrent.futures import ThreadPoolExecutor
    w = synth.NC4096
    freqs, dms = w.freqs(), w.dms()
    peaks, src = _peaks()
    gen = torch.Generator(device=dev).manual_seed(500)
    data = [[torch.randn((w.chunk, w.nchan), generator=gen, device=dev).mul_(16).add_(128).round_().clamp_(0, 255)
             .to(torch.uint8) for _ in range(2)] for _ in range(nbeams)]
    fill = int(np.ceil(4.148808e3 * w.dm_max * (freqs.min() ** -2 - freqs.max() ** -2) / synth.NC_DT / w.chunk)) + 1
    bpu = w.nchan / w.ndm + 4.0
    out = {"beams": nbeams, "nchan": w.nchan, "ndm": w.ndm, "chunk": w.chunk, "branching": w.branching}
    for name, m in (("graded", 1), ("float", 2)):
        t0 = time.perf_counter()
        with ThreadPoolExecutor(max_workers=min(nbeams, os.cpu_count() or 1)) as ex:
            plans = list(ex.map(lambda _: g.Plan(freqs, synth.NC_DT, dms, w.branching, m,
                                                 g.options(m, max_chunk=w.chunk), bind=False), range(nbeams)))
        build_s = time.perf_counter() - t0
        for p in plans:
            p.bind(device=dev)
        # one beam alone: tree time per steady chunk
        p0 = plans[0]
        for k in range(fill):
            p0.execute(data[0][k % 2])
        p0.profile(True)
        p0.profile_read()
        for k in range(4):
            p0.execute(data[0][k % 2])
        prof = p0.profile_read()
        p0.profile(False)
        tms = prof["tree"][0] / max(prof["tree"][1], 1)
        ach = bpu * w.chunk * w.ndm / (tms / 1e3) / 1e9
        row = {"plan_build_s": round(build_s, 2), "tree_ms_per_chunk": round(tms, 4),
               "tree_gdm_samples_per_s": round(w.chunk * w.ndm / (tms / 1e3) / 1e9, 2),
               "roofline": {"bound": "hbm", "achieved": ach, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                            "frac": ach / peaks["hbm_gbs"], "peak_source": src,
                            "algorithmic_bytes_per_dm_sample": bpu},
               "stage_ms_per_chunk": {k: round(v[0] / max(v[1], 1), 4) for k, v in prof.items()}}
        sweep = {}
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for k in (1, 2, 4, 8, 16):
            if k > nbeams:
                break
            for p in plans[:k]:
                p.bind(device=dev)
            batch = g.Batch(plans[:k])
            for s in range(fill):
                batch.execute([data[i][s % 2] for i in range(k)])
            torch.cuda.synchronize(dev)
            ev0.record()
            steps = 4
            for s in range(steps):
                batch.execute([data[i][s % 2] for i in range(k)])
            ev1.record()
            torch.cuda.synchronize(dev)
            ms = ev0.elapsed_time(ev1) / steps
            sweep[str(k)] = {"ms_per_step": round(ms, 3),
                             "gdm_samples_per_s": round(k * w.chunk * w.ndm / (ms / 1e3) / 1e9, 2),
                             "ring_mb_resident": round(k * w.nchan * p0.stats().ring_words * 4 / 1e6, 1)}
            for p in plans[:k]:
                p.candidates(check=False)
            del batch
        row["l2_residency_sweep"] = sweep
        out[name] = row
        del plans
        torch.cuda.empty_cache()
    out["note"] = ("random-noise beams (throughput only; parity of this shape is tests/test_gpu_fullsize.py); "
                   "graded saturates at N = 255 at 4096 channels; ring_mb_resident = one copy of every beam's "
                   "bit ring")
    return out


def zfloat_rate(g, args, dev, dchunks, freqs, dms):
    """Labelled-payload Mode C (precision study) on the same beam: the tree with FP16 and with
    FP32 partial-sum storage, timed per chunk by the stage events (plane only)."""
    import torch
    out = {}
    steps = max(1, min(args.steps, 3))
    for name, flag in (("fp16", g.FLAG_FP16_PARTIALS), ("fp32", 0)):
        p = g.Plan(freqs, synth.NC_DT, dms, BRANCHING, g.MODE_ZFLOAT,
                   g.options(g.MODE_ZFLOAT, max_chunk=W.chunk, flags=flag), device=dev)
        for _ in range(max(args.warmup, 1)):
            for c in dchunks:
                p.execute(c)
        p.profile(True)
        p.profile_read()
        for _ in range(steps):
            for c in dchunks:
                p.execute(c)
        prof = p.profile_read()
        p.profile(False)
        tms = prof["tree"][0] / max(prof["tree"][1], 1)
        ems = prof["encode"][0] / max(prof["encode"][1], 1)
        es = 2 if flag else 4
        bpu = W.nchan / W.ndm * es + 4.0  # payload ring read once per DM tile set + FP32 plane written
        peaks, src = _peaks()
        ach = bpu * W.chunk * W.ndm / (tms / 1e3) / 1e9
        # the reads of a tree that adds every channel for every DM, es bytes per (DM, sample, channel),
        # against SMs x 128 bytes per clock at the maximum SM clock (summing shared leaf patterns
        # once reads less: the fraction compares forms, it is not a share of the pipe)
        props = torch.cuda.get_device_properties(dev)
        smem_peak = props.multi_processor_count * 128 * float(peaks.get("sm_max_mhz") or 2070.0) * 1e6 / 1e9
        smem_ach = W.nchan * es * W.chunk * W.ndm / (tms / 1e3) / 1e9
        out[name] = {"tree_ms_per_chunk": round(tms, 4), "encode_ms_per_chunk": round(ems, 4),
                     "tree_gdm_samples_per_s": round(W.chunk * W.ndm / (tms / 1e3) / 1e9, 2),
                     "roofline": {"bound": "hbm", "achieved": ach, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                                  "frac": ach / peaks["hbm_gbs"], "peak_source": src,
                                  "algorithmic_bytes_per_dm_sample": bpu, "kernel": "k_tree_zs"},
                     "roofline_smem": {"bound": "smem", "achieved": smem_ach, "peak": smem_peak, "unit": "GB/s",
                                       "frac": smem_ach / smem_peak, "kernel": "k_tree_zs",
                                       "peak_source": f"derived: {props.multi_processor_count} SMs x 128 B/clock x "
                                                      "max SM clock",
                                       "algorithmic_bytes_per_dm_sample": W.nchan * es}}
    return out


SIFTER_FLOPS = 2 * (16384 * 16 * 9 + 4096 * 32 * 144 + 1024 * 64 * 288 + 16384 * 128)  # per snippet, forward


def sifter_rate(g, args, dev):
    """Learned sifter: BF16 tensor-core inference at batch 4096 and training steps at batch
    256 (CUDA events), and a short train/evaluate run on pipeline-made snippets comparing it
    with the plain S/N >= 7 sifter at equal false-alarm rate."""
    import torch
    from paper_2606_15361_gb300 import sifter_data as sd
    gen = torch.Generator(device=dev).manual_seed(7)
    xb = torch.randn((4096, 64, 256), generator=gen, device=dev)
    inf = g.Sifter(max_batch=4096, training=False, seed=1, device=dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(3):
        inf.forward(xb)
    ev0.record()
    for _ in range(10):
        inf.forward(xb)
    ev1.record()
    torch.cuda.synchronize(dev)
    inf_ms = ev0.elapsed_time(ev1) / 10
    tr_sf = g.Sifter(max_batch=256, training=True, seed=1, device=dev)
    yb = (torch.rand(256, generator=gen, device=dev) < 0.5).float()
    for _ in range(3):
        tr_sf.train_step(xb[:256], yb, 1e-4)
    ev0.record()
    for _ in range(20):
        tr_sf.train_step(xb[:256], yb, 1e-4)
    ev1.record()
    torch.cuda.synchronize(dev)
    step_ms = ev0.elapsed_time(ev1) / 20
    del inf, tr_sf
    tr = sd.concat([sd.make_run(3000 + i, n_burst=96, device=dev) for i in range(30)])
    te = sd.concat([sd.make_run(93000 + i, n_burst=96, device=dev) for i in range(10)])
    sf = g.Sifter(max_batch=256, training=True, seed=2, device=dev)
    sd.train(sf, tr, epochs=5, batch=256, lr=5e-4)
    cmp = sd.compare(sd.logits(sf, te.x, 256), te)
    peaks, src = _peaks()
    tfl = SIFTER_FLOPS * 4096 / (inf_ms / 1e3) / 1e12
    return {"roofline": {"bound": "tensor", "achieved": tfl, "peak": peaks["bf16_tflops"], "unit": "TFLOP/s",
                         "frac": tfl / peaks["bf16_tflops"], "peak_source": src,
                         "kernel": "sifter forward (k_gemm + layer kernels), batch 4096",
                         "algorithmic_flops_per_snippet": SIFTER_FLOPS},
            "infer_batch": 4096, "infer_ms_per_batch": round(inf_ms, 3),
            "infer_snippets_per_s": round(4096 / (inf_ms / 1e3), 1),
            "infer_tflops": round(SIFTER_FLOPS * 4096 / (inf_ms / 1e3) / 1e12, 2),
            "train_batch": 256, "train_ms_per_step": round(step_ms, 3),
            "train_snippets_per_s": round(256 / (step_ms / 1e3), 1),
            "quick_eval": {"train_snippets": int(len(tr.label)), "test_snippets": int(len(te.label)),
                           "far_plain": round(cmp["far_plain"], 4), "miss_plain": round(cmp["miss_plain"], 4),
                           "far_learned": round(cmp["far_learned"], 4), "miss_learned": round(cmp["miss_learned"], 4)},
            "note": "quick_eval: 30 synthetic beam runs, 5 epochs; the full 200k-snippet run is "
                    "paper_2606_15361_gb300/sifter_train.py"}


def multibeam_setup(g, dev, nbeams=48, seed=11, branching=None, steps_tune=2):
    """The 48 ragged beams of the many-beam row: configs, data (two chunks per beam) and B."""
    import torch
    from paper_2606_15361_gb300 import autotune
    rng = np.random.default_rng(seed)
    f = synth.channel_freqs(1024)
    tune = None
    shape = {"tree_warps": 0, "tree_round": 0}
    if branching is None:
        tune = autotune.autotune(f, synth.NC_DT, synth.dm_grid(2048, 2000.0), g.MODE_FLOAT, 16384,
                                 branching=(8, 2, 4, 16), cluster=(4,), steps=steps_tune, device=dev)
        branching = tune["branching"]
        shape = {"tree_warps": tune["tree_warps"], "tree_round": tune["tree_round"]}
    cfgs = [(int(rng.integers(512, 4097)), float(rng.uniform(500.0, 3000.0)), int(rng.integers(4, 33)) * 1024)
            for _ in range(nbeams)]
    gen = torch.Generator(device=dev).manual_seed(seed)
    data = [[torch.randn((ch, 1024), generator=gen, device=dev).mul_(16).add_(128).round_().clamp_(0, 255)
             .to(torch.uint8) for _ in range(2)] for _, _, ch in cfgs]
    fill = max((p_d + ch - 1) // ch for p_d, ch in
               ((int(2.0 + 4.148808e3 * dmx * (f.min() ** -2 - f.max() ** -2) / synth.NC_DT), ch) for _, dmx, ch in cfgs))
    return f, cfgs, data, branching, tune, fill, shape


def multibeam_rate(g, args, dev, nbeams=48, seed=11):
    """Ragged beams in one step: 48 beams of 1024 channels, each with its own DM grid
    (512-4096 trials to a max DM of 500-3000) and chunk length (4096-32768 samples), float
    mode, branching from the autotuner. Times one step of all beams run plan by plan, as a
    batch (grouped tree launches), and as a batch replayed through a CUDA graph."""
    import torch
    f, cfgs, data, B, tune, fill, shape = multibeam_setup(g, dev, nbeams, seed)

    def make():
        return [g.Plan(f, synth.NC_DT, synth.dm_grid(nd, dmx), B, g.MODE_FLOAT,
                       g.options(g.MODE_FLOAT, max_chunk=ch, **shape), device=dev) for nd, dmx, ch in cfgs]

    steps = max(2, min(args.steps, 5))
    out = {"beams": nbeams,
           "autotune": {"branching": B, "tree_warps": tune["tree_warps"], "tree_round": tune["tree_round"],
                        "significant": tune["significant"],
                        "trials": [(t["branching"], t["tree_warps"], t["tree_round"], round(t["ms_per_chunk"], 4),
                                    round(t["spread_ms"], 4)) for t in tune["trials"]],
                        "note": "trial = (B, warps per tree CTA, channels per staging round, median pipeline ms per "
                                "chunk, spread over 3 repeats); a pick replaces the default (B = 8, 8 warps, 128) "
                                "only when it beats it by more than both spreads"}}
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for name in ("per_beam", "batch", "batch_graph"):
        plans = make()
        batch = g.Batch(plans, graph=(name == "batch_graph")) if name != "per_beam" else None

        def step(k):
            if batch is None:
                for i, p in enumerate(plans):
                    p.execute(data[i][k % 2])
            else:
                batch.execute([data[i][k % 2] for i in range(nbeams)])

        for k in range(fill + 2):
            step(k)
        for p in plans:
            p.candidates(check=False)
        torch.cuda.synchronize(dev)
        launches0 = sum(p.stats().kernel_launches for p in plans)
        ev0.record()
        for k in range(steps):
            step(k)
        ev1.record()
        torch.cuda.synchronize(dev)
        ms = ev0.elapsed_time(ev1) / steps
        launches = (sum(p.stats().kernel_launches for p in plans) - launches0) // steps
        out[name] = {"ms_per_step": round(ms, 3), "kernels_per_step": int(launches)}
        del batch, plans
        torch.cuda.empty_cache()
    units = sum(nd * ch for nd, _, ch in cfgs)
    best = min(out[k]["ms_per_step"] for k in ("batch", "batch_graph"))
    shortest = min(ch for _, _, ch in cfgs) * synth.NC_DT * 1e3
    out.update({"dm_samples_per_step": units, "gdm_samples_per_s_batch_graph":
                round(units / (out["batch_graph"]["ms_per_step"] / 1e3) / 1e9, 2),
                "shortest_chunk_ms": round(shortest, 1),
                "realtime_margin": round(shortest / best, 1),
                "note": "all beams advance one chunk per step; the step must finish within the shortest "
                        "chunk's duration for every beam to keep up; realtime_margin = that duration / step time"})
    return out


def run_gpu(args, rank, world, local_rank):
    import torch
    import paper_2606_15361_gb300 as g
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    host_chunks = [W.chunk_data(i) for i in range(W.nchunks)]
    dchunks = [torch.from_numpy(c).to(dev) for c in host_chunks]                  # 268 MB > L2
    pinned = [torch.from_numpy(c).pin_memory() for c in host_chunks]
    freqs, dms = W.freqs(), W.dms()
    plans = {name: g.Plan(freqs, synth.NC_DT, dms, BRANCHING, m, g.options(m, max_chunk=W.chunk), device=dev)
             for name, m in MODES}
    stream = torch.cuda.current_stream(dev)
    # the three modes are independent, so by default each plan runs on its own stream and one
    # mode's small matched-filter and candidate kernels overlap another mode's tree
    mstreams = {name: torch.cuda.Stream(dev) for name, _ in MODES}

    def step(host: bool, concurrent: bool):
        if concurrent:
            ev = torch.cuda.Event()
            ev.record(stream)
            for name, _ in MODES:
                mstreams[name].wait_event(ev)
        for name, _ in MODES:
            p = plans[name]
            st = mstreams[name] if concurrent else stream
            for i in range(W.nchunks):
                if host:
                    p.execute_host(pinned[i], stream=st)
                else:
                    p.execute(dchunks[i], stream=st)
        if concurrent:
            for name, _ in MODES:
                done = torch.cuda.Event()
                done.record(mstreams[name])
                stream.wait_event(done)

    def sync():
        torch.cuda.synchronize(dev)
        if dist:
            dist.barrier()

    concurrent = not args.sequential
    # warm-up (also fills the rings: from then on every chunk emits W.chunk samples per row)
    for _ in range(max(args.warmup, 1)):
        step(False, concurrent)
    for p in plans.values():
        p.candidates(check=False)
    sync()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    # pass 1, modes in sequence on one stream, per-stage CUDA events: every launch's duration
    # is its own (the roofline and the per-mode stage times)
    for p in plans.values():
        p.profile(True)
        p.profile_read()
    sync()
    ev0.record(stream)
    for _ in range(args.steps):
        step(False, False)
    ev1.record(stream)
    sync()
    ms_seq = ev0.elapsed_time(ev1)
    prof = {n: p.profile_read() for n, p in plans.items()}
    for p in plans.values():
        p.profile(False)
    for p in plans.values():
        p.candidates(check=False)

    # pass 2, the headline: the three modes on their own streams
    launches0 = {n: p.stats().kernel_launches for n, p in plans.items()}
    clocks = ClockSampler(local_rank)
    clocks.start()
    sync()
    ev0.record(stream)
    for _ in range(args.steps):
        step(False, concurrent)
    ev1.record(stream)
    sync()
    ms_dev = ev0.elapsed_time(ev1)
    clk = clocks.stop()
    launches = sum(p.stats().kernel_launches - launches0[n] for n, p in plans.items())
    ncands = sum(len(p.candidates(check=False)[0]) for p in plans.values())

    # end to end: pinned host chunks copied inside the C-ABI call, candidates read back
    for p in plans.values():
        p.candidates(check=False)
    sync()
    t0 = time.perf_counter()
    ev0.record(stream)
    d2h = 0
    for _ in range(args.steps):
        step(True, concurrent)
        for p in plans.values():
            c, _ = p.candidates(check=False)
            d2h += c.nbytes + 8
    ev1.record(stream)
    sync()
    ms_e2e = max(ev0.elapsed_time(ev1), 1e3 * (time.perf_counter() - t0))

    extras = rank == 0 and not args.main_only
    mr = multirate_rate(g, args, dev, stream, dchunks, freqs, dms) if extras else None
    bsw = branching_sweep(g, args, dev, dchunks, freqs, dms) if extras else None
    c5 = stress_rate(g, args, dev) if extras and not args.no_stress else None
    zf = zfloat_rate(g, args, dev, dchunks, freqs, dms) if extras else None
    sft = sifter_rate(g, args, dev) if extras and not args.no_sifter else None
    mb = multibeam_rate(g, args, dev) if extras and not args.no_multibeam else None

    per_step = len(MODES) * W.nchunks * W.chunk * W.ndm   # DM-samples per step per GPU
    ms_dev, ms_e2e, ms_seq = reduce_max([ms_dev, ms_e2e, ms_seq], dist, dev)
    value = whole_job_rate(per_step, args.steps, world, ms_dev)
    e2e = whole_job_rate(per_step, args.steps, world, ms_e2e)
    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return None

    peaks, src = _peaks()
    tree_ms = sum(prof[n]["tree"][0] for n in prof)
    tree_n = sum(prof[n]["tree"][1] for n in prof)
    tree_launch_ms = tree_ms / max(tree_n, 1)
    units = W.chunk * W.ndm
    achieved = TREE_BYTES_PER_DM_SAMPLE * units / (tree_launch_ms / 1e3) / 1e9
    per_mode = {}
    # the tree's algorithmic ALU work per DM-sample (see ALU_LANES_PER_SM_CYCLE) against the
    # ALU-pipe ceiling of this GPU at the maximum SM clock
    props = torch.cuda.get_device_properties(dev)
    sm_max = float(clk.get("sm_max_mhz") or peaks.get("sm_max_mhz") or 2070.0)
    alu_peak = props.multi_processor_count * ALU_LANES_PER_SM_CYCLE * sm_max * 1e6 / 1e9  # Gop/s
    adds = {n: (9.0 * W.nchan / 128.0 if n == "binary" else 3.0 * W.nchan / 32.0) for n in prof}
    for n in prof:
        st = {k: round(v[0] / max(v[1], 1), 4) for k, v in prof[n].items()}
        tms = prof[n]["tree"][0] / max(prof[n]["tree"][1], 1)
        per_mode[n] = {"stage_ms_per_chunk": st,
                       "tree_gdm_samples_per_s": round(units / (tms / 1e3) / 1e9, 2),
                       "tree_hbm_frac": round(TREE_BYTES_PER_DM_SAMPLE * units / (tms / 1e3) / 1e9 /
                                              peaks["hbm_gbs"], 4),
                       "tree_alu_frac": round(adds[n] * units / (tms / 1e3) / 1e9 / alu_peak, 4),
                       # the matched filter reads the int32 plane once: 4 B per DM-sample
                       "mf_hbm_frac": round(4.0 * units / (prof[n]["mf"][0] / max(prof[n]["mf"][1], 1) / 1e3) / 1e9 /
                                            peaks["hbm_gbs"], 4),
                       "pipeline_gdm_samples_per_s": round(units / (sum(v[0] for v in prof[n].values()) /
                                                                    max(prof[n]["tree"][1], 1) / 1e3) / 1e9, 2)}
    adds_mean = sum(adds.values()) / max(len(adds), 1)
    traffic = _traffic_from_profile(_tree_source_hash())
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        cpu = oracle_sample(host_chunks[:3])
        if not args.main_only:
            cpu["rows"] = oracle_rows_sample(host_chunks)
    realtime_beams = e2e / (W.ndm / synth.NC_DT) / len(MODES)
    return {
        "metric": "DM-trial samples/s", "value": value, "unit": "DM-samples/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_dev / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u1/int32",
        "data": DATA_NOTE,
        "config": {"workload": "nc1024_2048dm: 1024 ch 400-416 MHz, dt 0.138 ms, 2048 DMs 0-2000 pc/cm3, "
                               "16 x 16384-sample chunks per step, B=8, modes binary+graded+float (Table S1)",
                   "branching": BRANCHING, "chunk": W.chunk, "chunks_per_step": W.nchunks,
                   "l2": "inputs larger than L2 (16 chunks = 268 MB uint8 per step, 129 MB L2)",
                   "parallelism": f"beam replicas x{world}",
                   "streams": "one per mode" if concurrent else "one"},
        "gpu_launches": int(launches),
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                     "frac": achieved / peaks["hbm_gbs"], "traffic": traffic,
                     "kernel": "k_snd (SND tree, all modes, average launch, sequential pass)",
                     "peak_source": src, "algorithmic_bytes_per_dm_sample": TREE_BYTES_PER_DM_SAMPLE},
        "roofline_alu": {"bound": "alu", "achieved": adds_mean * units / (tree_launch_ms / 1e3) / 1e9,
                         "peak": alu_peak, "unit": "Gop/s",
                         "frac": adds_mean * units / (tree_launch_ms / 1e3) / 1e9 / alu_peak,
                         "kernel": "k_snd (SND tree, all modes, average launch, sequential pass)",
                         "algorithmic_ops_per_dm_sample": adds_mean,
                         "peak_source": (f"derived: {props.multi_processor_count} SMs x 4 sub-partitions x 16 ALU lanes "
                                         f"(LOP3/SHF) x {sm_max:.0f} MHz; ops = funnel shifts + carry-save adders "
                                         "(float/graded 3 N_f/32, binary 9 N_f/128 per DM-sample)")},
        "per_mode": per_mode,
        "sequential_pass": {"value": whole_job_rate(per_step, args.steps, world, ms_seq), "unit": "DM-samples/s",
                            "ms_per_step": ms_seq / args.steps,
                            "note": "modes in sequence on one stream with per-stage events; the roofline "
                                    "and per_mode stage times come from this pass"},
        "e2e": {"value": e2e, "unit": "DM-samples/s",
                "h2d_bytes_per_step": len(MODES) * W.nchunks * W.chunk * W.nchan,
                "d2h_bytes_per_step": int(d2h / max(args.steps, 1))},
        "realtime_beams_per_mode": realtime_beams,
        "multirate": mr,
        "branching_sweep": bsw,
        "stress_nc4096": c5,
        "zfloat_precision_study": zf,
        "learned_sifter": sft,
        "multibeam": mb,
        "candidates_in_timed_steps": ncands,
        "cpu_baseline": cpu,
        "clocks": clk,
    }


def drive(mode_name: str, nchunks: int, branching: int):
    """Run one plan of the workload over `nchunks` chunks, untimed (for profiler captures:
    the tree kernel's second launch is the first steady-state chunk). Modes beyond the three
    tree modes: zfloat / zfloat16 (labelled payload, FP32 / FP16 partial sums), sifter (the
    learned sifter: forward passes at batch 512, then training steps at batch 256; about 2 GB
    of device memory, small enough for a full profiler capture)."""
    import torch
    import paper_2606_15361_gb300 as g
    if mode_name == "batch48":
        dev = torch.device("cuda", 0)
        f, cfgs, data, B, _, fill, shape = multibeam_setup(g, dev, branching=branching)
        plans = [g.Plan(f, synth.NC_DT, synth.dm_grid(nd, dmx), B, g.MODE_FLOAT,
                        g.options(g.MODE_FLOAT, max_chunk=ch, **shape), device=dev) for nd, dmx, ch in cfgs]
        batch = g.Batch(plans)
        for k in range(fill + nchunks):
            batch.execute([data[i][k % 2] for i in range(len(plans))])
        torch.cuda.synchronize()
        print(json.dumps({"drive": mode_name, "steps": fill + nchunks, "branching": B}))
        return
    if mode_name == "sifter":
        gen = torch.Generator(device="cuda").manual_seed(7)
        x = torch.randn((512, 64, 256), generator=gen, device="cuda")
        y = (torch.rand(512, generator=gen, device="cuda") < 0.5).float()
        inf = g.Sifter(max_batch=512, training=False, seed=1)
        for _ in range(nchunks):
            inf.forward(x)
        tr = g.Sifter(max_batch=256, training=True, seed=1)
        for _ in range(nchunks):
            tr.train_step(x[:256], y[:256], 1e-4)
        tr.status()
        print(json.dumps({"drive": mode_name, "passes": nchunks}))
        return
    if mode_name in ("zfloat", "zfloat16"):
        chunks = [torch.from_numpy(W.chunk_data(i)).cuda() for i in range(nchunks)]
        flag = g.FLAG_FP16_PARTIALS if mode_name == "zfloat16" else 0
        plan = g.Plan(W.freqs(), synth.NC_DT, W.dms(), branching, g.MODE_ZFLOAT,
                      g.options(g.MODE_ZFLOAT, max_chunk=W.chunk, flags=flag))
        for c in chunks:
            plan.execute(c)
        torch.cuda.synchronize()
        print(json.dumps({"drive": mode_name, "chunks": nchunks, "branching": branching}))
        return
    m = dict(MODES)[mode_name]
    chunks = [torch.from_numpy(W.chunk_data(i)).cuda() for i in range(nchunks)]
    plan = g.Plan(W.freqs(), synth.NC_DT, W.dms(), branching, m, g.options(m, max_chunk=W.chunk))
    for c in chunks:
        plan.execute(c)
    torch.cuda.synchronize()
    _, rc = plan.candidates(check=False)
    print(json.dumps({"drive": mode_name, "chunks": nchunks, "branching": branching, "status": rc}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sifter", action="store_true", help="skip the learned-sifter measurements")
    ap.add_argument("--no-multibeam", action="store_true", help="skip the 48-beam batch measurements")
    ap.add_argument("--no-stress", action="store_true", help="skip the 16-beam 4096-channel stress measurements")
    ap.add_argument("--sequential", action="store_true",
                    help="headline pass with the three modes in sequence on one stream (default: own streams)")
    ap.add_argument("--main-only", action="store_true",
                    help="only the headline workload: no multi-rate, labelled-payload, sifter or multi-beam parts")
    ap.add_argument("--drive", choices=[m for m, _ in MODES] + ["zfloat", "zfloat16", "sifter", "batch48"],
                    help="profiling driver: one plan (or the sifter), no timing")
    ap.add_argument("--chunks", type=int, default=3)
    ap.add_argument("--branching", type=int, default=BRANCHING)
    args = ap.parse_args()
    if args.drive:
        drive(args.drive, args.chunks, args.branching)
        return
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", str(args.gpus if args.gpus == 1 else 1)))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        res = run_reference(args, rank, world)
    else:
        res = run_gpu(args, rank, world, local_rank)
    if res is not None and rank == 0:
        print(json.dumps(res), flush=True)


if __name__ == "__main__":
    main()
