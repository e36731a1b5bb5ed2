#!/usr/bin/env python
"""Benchmark of the adaptive histogram stream on GB300.

Workload (one step): a 1 GiB uint8 stream of clamp(round(N(128, 8))) pixels
(the X-ray-like peaked distribution) cut into 64 chunks of 16 MiB, pushed
through the chunked stream with the adaptive kernel, the binning pattern of
each chunk refreshed on the device from the previous chunk's histogram, the
degeneracy switch evaluated and the totals accumulated (every step of the hot
path).  Inputs are generated on the device and resident in HBM before the
timed region; at 1 GiB they are larger than the 129 MB L2.

Prints one JSON line (rank 0).  `--impl reference` times the CPU oracle on a
bounded sample of the same workload instead.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

MiB = 1 << 20
CHUNK = 16 * MiB
METRIC = "input GB/s (% of HBM peak), adaptive vs plain kernel; p50/p99 request latency"
UNIT = "GB/s"
CPU_SAMPLE_SECONDS = 10.0
STREAM_MAX_BATCH = 1024  # chunks per launch of the stream kernels
SERVE_RATES = (2000, 5000, 10000, 20000, 50000)  # requests per second
SERVE_SECONDS = 0.5  # of arrivals per rate
CPU_THREADS_SECONDS = 3.0  # of the threaded oracle count


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="native", choices=["native", "reference"])
    ap.add_argument("--chunks", type=int, default=64, help="chunks of 16 MiB per step (64 = 1 GiB)")
    ap.add_argument("--profile", action="store_true",
                    help="headline stream only: no clock settling, extras, end-to-end or CPU legs (for ncu)")
    ap.add_argument("--profile-part", default=None,
                    choices=["serving", "batch", "ablation", "table2", "auto", "budget960", "smallchunks",
                             "budgets", "regimes"],
                    help="run only one other workload once, for ncu: the serving capacity replay "
                         "(4000 requests), the 4096-image batch, 256 MiB cases of Table 1 and Table 2, "
                         "the degenerate workload through an AUTO stream, the N(128, 8) stream at "
                         "960 slots, or 256 MiB of it in 64 KiB chunks")
    return ap.parse_args()


def workload_config(chunks):
    return {
        "workload": "stream of %d MiB uint8 in 16 MiB chunks, clamp(round(N(128, sigma=8))), adaptive kernel, "
                    "binning pattern refreshed per chunk on the device" % (chunks * 16),
        "bytes_per_step": chunks * CHUNK,
        "chunk_bytes": CHUNK,
        "chunks": chunks,
        "budget": 8192,
        "theta_milli": 450,
        "pushes": "HIST_OVERLAP_PUSHES: the chunks are resident and complete before the timed region, so a "
                  "push's counting launch may start reading while the previous push finishes (without the "
                  "flag a launch reads nothing before the work before it completes: extras.adaptive_stream_default_gbs)",
        "l2": "inputs larger than L2 (1 GiB vs 129 MB); no flush needed" if chunks * CHUNK > 256 * MiB
        else "inputs smaller than 2x L2: numbers include L2 reuse",
    }


def dist_env():
    from paper_1011_0235_gb300 import shard

    return shard.env()


# ------------------------------------------------------------- clocks ----

class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled every 50 ms."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None
        self.t0 = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                 "-lms", "50"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        self.t0 = time.time()

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.06)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append(parts)
            except ValueError:
                pass
        os.unlink(self.path)
        if not rows:
            return None

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None

        sm = [num(r[1]) for r in rows if num(r[1]) is not None]
        mx = [num(r[2]) for r in rows if num(r[2]) is not None]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            for name, val in zip(names, r[5:9]):
                if val.strip().lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(rows),
                "power_w_max": max([num(r[3]) for r in rows if num(r[3]) is not None] or [0])}


# ------------------------------------------------------------ helpers ----

def measured_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        return None


# The sources a kernel is compiled from (its translation unit and headers).
KERNEL_SOURCES = {
    "batch_flat_kernel": ["paper_1011_0235_gb300/csrc/hist_stream.cu", "paper_1011_0235_gb300/csrc/hist_device.cuh",
                          "paper_1011_0235_gb300/csrc/hist_internal.h", "paper_1011_0235_gb300/csrc/hist_plan.h",
                          "include/hist.h"],
}


def sources_hash(kernel):
    """Hash of the kernel's sources with comments and whitespace left out:
    the recorded traffic depends on the code, not on its documentation."""
    import re

    h = hashlib.sha256()
    for f in KERNEL_SOURCES[kernel]:
        text = open(os.path.join(ROOT, f), encoding="utf-8").read()
        text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
        text = re.sub(r"//[^\n]*", " ", text)
        h.update(f.encode())
        h.update(" ".join(text.split()).encode())
    return h.hexdigest()[:16]


def recorded_traffic(kernel):
    """DRAM bytes per launch from the committed ncu summary, if it was taken on
    the kernel's current sources."""
    try:
        rec = json.load(open(os.path.join(ROOT, "profiles", "traffic.json")))
    except (OSError, ValueError):
        return None
    k = rec.get(kernel)
    if not k or k.get("sources_hash") != sources_hash(kernel):
        return None
    return k.get("dram_bytes_per_launch")


def gen_workload_device(torch, synth, chunks, seed, thr_fn, first_chunk=0):
    """Chunks first_chunk .. first_chunk + chunks - 1 of the synthetic stream
    (a rank's own slice of one long stream)."""
    x = torch.empty(chunks * CHUNK, dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for c in range(chunks):
        g = first_chunk + c
        synth.device_fill(x.data_ptr() + c * CHUNK, CHUNK, thr_fn(g), seed, g * CHUNK, s)
    torch.cuda.synchronize()
    return x


def time_steps(torch, step, warmup, steps, barrier=None):
    for _ in range(warmup):
        step()
    torch.cuda.synchronize()
    if barrier:
        barrier()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(steps):
        step()
    e1.record()
    torch.cuda.synchronize()
    if barrier:
        barrier()
    return e0.elapsed_time(e1) / 1e3  # seconds


def cpu_oracle_rate(host_chunks, seconds):
    """Time the oracle's stream (hist + switch + pattern per chunk) on host cores
    over the given chunks, repeated until `seconds` have passed."""
    import oracle

    oracle.lib()
    done = 0
    t0 = time.perf_counter()
    while True:
        so = oracle.StreamOracle(8192, mode=oracle.MODE_ADAPTIVE)
        for ch in host_chunks:
            so.push(ch)
            done += ch.size
        el = time.perf_counter() - t0
        if el >= seconds:
            return done / el / 1e9, done, el


def cpu_oracle_threads_rate(buf, seconds, threads):
    """The oracle's counting loop on `threads` host threads at once: each
    thread counts its own contiguous slice of `buf` into a private u64[256]
    (ctypes releases the GIL during the call) and the slices' histograms are
    summed; repeated until `seconds` have passed.  Returns the rate, the bytes
    counted, the time and the summed histogram of one pass."""
    from concurrent.futures import ThreadPoolExecutor
    import numpy as np
    import oracle

    lib = oracle.lib()
    n = buf.size
    cuts = [n * k // threads for k in range(threads + 1)]
    hs = [np.zeros(256, np.uint64) for _ in range(threads)]

    def work(k):
        lib.oracle_hist_u64(buf.ctypes.data + cuts[k], cuts[k + 1] - cuts[k], hs[k].ctypes.data)

    done = 0
    t0 = time.perf_counter()
    with ThreadPoolExecutor(threads) as ex:
        while True:
            list(ex.map(work, range(threads)))
            total = np.sum(hs, axis=0, dtype=np.uint64)
            done += n
            el = time.perf_counter() - t0
            if el >= seconds:
                return done / el / 1e9, done, el, total


def host_fed_extras(torch, hl, hx, chunks, steps):
    """Sec. III.B's host-fed stream on this machine (Table 3's question: how
    much of the transfer the kernels hide): GB/s of the adaptive stream fed
    from pinned host memory, sequentially (each chunk copied, then counted,
    on one CUDA stream) and pipelined (hist_stream_push_host with 2, 3 and 4
    staging buffers attached, which pinned chunks do not use: the counting
    kernels read them over the host link)."""
    res = {}
    d = torch.empty(CHUNK, dtype=torch.uint8, device="cuda")
    st = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE)

    def seq_step():
        for c in range(chunks):
            d.copy_(hx[c * CHUNK:(c + 1) * CHUNK], non_blocking=True)
            st.push(d)
        st.flush()

    el = time_steps(torch, seq_step, 2, steps)
    res["sequential_gbs"] = round(chunks * CHUNK * steps / el / 1e9, 2)
    st.close()
    del d
    for depth in (2, 3, 4):
        st = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE)
        st.attach_staging(CHUNK, depth)

        def pipe_step():
            for c in range(chunks):
                st.push_host(hx.data_ptr() + c * CHUNK, CHUNK)
            st.flush()

        el = time_steps(torch, pipe_step, 2, steps)
        res["staging_depth_%d_gbs" % depth] = round(chunks * CHUNK * steps / el / 1e9, 2)
        st.close()
    # Figs. 3 and 4: the pipelined time over the sequential time as the
    # number of chunks grows (4 MiB chunks, 1 .. 256 of them), each step
    # timed alone (synchronised before and after) so that steps do not overlap
    c4 = 4 << 20
    sweep = {"chunk_bytes": c4, "chunks": [k for k in (1, 4, 16, 64, 256) if k * c4 <= hx.numel()],
             "pipelined_over_sequential": []}
    d4 = torch.empty(c4, dtype=torch.uint8, device="cuda")

    def alone(step, reps):
        step()
        tot = 0.0
        for _ in range(reps):
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record()
            step()
            e1.record()
            torch.cuda.synchronize()
            tot += e0.elapsed_time(e1)
        return tot / reps

    for k in sweep["chunks"]:
        s1 = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE)

        def seq_k(s1=s1, k=k):
            for c in range(k):
                d4.copy_(hx[c * c4:(c + 1) * c4], non_blocking=True)
                s1.push(d4)
        t_seq = alone(seq_k, 5)
        s1.close()
        s2 = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE)
        s2.attach_staging(c4, 3)

        def pipe_k(s2=s2, k=k):
            for c in range(k):
                s2.push_host(hx.data_ptr() + c * c4, c4)
        t_pipe = alone(pipe_k, 5)
        s2.close()
        sweep["pipelined_over_sequential"].append(round(t_pipe / t_seq, 3))
    res["chunks_sweep"] = sweep
    return res


def batch_extras(torch, hl, synth, hbm, steps, autotune=True):
    """4096 images of uneven sizes in one graph-captured launch, with the
    autotuner's setting (or the default setting)."""
    import ctypes
    from paper_1011_0235_gb300 import _abi
    from synth import workloads
    images = workloads.batch_images(count=4096)
    bbytes = sum(im.n for im in images)
    bbuf = torch.empty(workloads.packed_bytes(images), dtype=torch.uint8, device="cuda")
    sq = torch.cuda.current_stream().cuda_stream
    for im in images:
        synth.device_fill(bbuf.data_ptr() + im.offset, im.n, im.thr, synth.SEED_BASE + 4, im.counter0, sq)
    bptrs = torch.tensor([bbuf.data_ptr() + im.offset for im in images], dtype=torch.int64, device="cuda")
    bsizes = torch.tensor([im.n for im in images], dtype=torch.int64, device="cuda")
    bout = torch.empty((len(images), 256), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    lib = hl.lib()
    best = _abi.BatchTuning()
    lib.hist_batch_tuning_init(ctypes.byref(best))
    if autotune:
        bms = ctypes.c_float()
        _abi.check("hist_batch_autotune", lib.hist_batch_autotune(bptrs.data_ptr(), bsizes.data_ptr(), len(images),
                                                                  bout.data_ptr(), 2, ctypes.byref(best),
                                                                  ctypes.byref(bms)))
    gexec = ctypes.c_void_p()
    _abi.check("hist_batch_capture", lib.hist_batch_capture(bptrs.data_ptr(), bsizes.data_ptr(), len(images),
                                                            bout.data_ptr(), ctypes.byref(best), ctypes.byref(gexec)))
    e5 = time_steps(torch, lambda: _abi.check("hist_batch_graph_launch", lib.hist_batch_graph_launch(
        gexec, torch.cuda.current_stream().cuda_stream)), 2 if autotune else 0, steps)
    lib.hist_batch_graph_destroy(gexec)
    out = {"batch_images": len(images), "batch_bytes": bbytes,
           "batch_graph_gbs": round(bbytes * steps / e5 / 1e9, 2),
           "batch_frac_of_hbm": round(bbytes * steps / e5 / 1e9 / hbm, 4),
           "batch_tuning": {"ctas_per_sm": best.ctas_per_sm, "unroll": best.unroll,
                            "small_bytes": best.small_bytes, "small_log2k": best.small_log2k}}
    if autotune:
        out["batch_regimes"] = regime_extras(torch, lib, _abi, images, bbuf, bptrs, bsizes, bout, hbm, steps)
        # the same batch with a third of the images given the degenerate law
        for k, im in enumerate(images):
            if k % 3 == 0:
                synth.device_fill(bbuf.data_ptr() + im.offset, im.n, synth.degenerate(90, 0.95), synth.SEED_BASE + 4,
                                  im.counter0, sq)
        torch.cuda.synchronize()
        out["batch_regimes_with_degenerate_third"] = regime_extras(torch, lib, _abi, images, bbuf, bptrs, bsizes,
                                                                   bout, hbm, steps)
    return out


def regime_extras(torch, lib, _abi, images, bbuf, bptrs, bsizes, bout, hbm, steps):
    """The batch tuned per distribution regime: the table the autotuner picks,
    each regime's images alone with that setting and with the default full
    table, and the whole batch as one graph (classification + counting)."""
    import ctypes
    names = ("degenerate", "peaked", "wide")
    reg = torch.empty(len(images), dtype=torch.uint8, device="cuda")
    best = _abi.BatchTable()
    lib.hist_batch_table_init(ctypes.byref(best))
    rep = _abi.RegimeReport()
    _abi.check("hist_batch_autotune_regimes", lib.hist_batch_autotune_regimes(
        bptrs.data_ptr(), bsizes.data_ptr(), len(images), bout.data_ptr(), reg.data_ptr(), 2, ctypes.byref(best),
        ctypes.byref(rep)))

    def lay(v):
        return "per_warp" if v == _abi.LAYOUT_PER_WARP else "k=%d" % (1 << v)

    table = {}
    for r, nm in enumerate(names):
        st = best.regime[r]
        b = rep.bytes[r]
        table[nm] = {"images": rep.images[r], "bytes": b, "layout": lay(st.layout),
                     "small_bytes": st.small_bytes, "small_layout": lay(st.small_layout) if st.small_bytes else None,
                     "gbs": round(b / rep.ms[r] / 1e6, 1) if rep.ms[r] > 0 else None,
                     "default_full_table_gbs": round(b / rep.ms_default[r] / 1e6, 1) if rep.ms_default[r] > 0 else None}
    bbytes = sum(im.n for im in images)
    g = ctypes.c_void_p()
    _abi.check("hist_batch_regimes_capture", lib.hist_batch_regimes_capture(
        bptrs.data_ptr(), bsizes.data_ptr(), len(images), bout.data_ptr(), reg.data_ptr(), ctypes.byref(best),
        ctypes.byref(g)))
    el = time_steps(torch, lambda: _abi.check("hist_batch_graph_launch", lib.hist_batch_graph_launch(
        g, torch.cuda.current_stream().cuda_stream)), 2, steps)
    lib.hist_batch_graph_destroy(g)
    return {"ctas_per_sm": best.ctas_per_sm, "unroll": best.unroll, "candidates_per_regime": rep.candidates,
            "regimes": table, "graph_gbs": round(bbytes * steps / el / 1e9, 2),
            "graph_frac_of_hbm": round(bbytes * steps / el / 1e9 / hbm, 4),
            "autotuner_batch_gbs": round(bbytes / rep.batch_ms / 1e6, 1),
            "autotuner_default_table_gbs": round(bbytes / rep.batch_default_ms / 1e6, 1)}


def ablation_extras(torch, hl, synth, hbm, steps=10, n=1 << 30):
    """Table 1 on this GPU: GB/s of the five cumulative kernel variants on
    n bytes (1 GiB) of uniform pixels (the paper's random input) and of N(128, 8), for
    the per-warp kernel, the adaptive kernel with the 960-slot default
    pattern (the paper's table) and with the full 8192-slot table."""
    from paper_1011_0235_gb300 import _abi
    lib = hl.lib()
    full = ([32 * b for b in range(256)], [5] * 256, 8192, 8192)
    pats = {"plain": None, "adaptive_960": hl.default_pattern(960),
            "adaptive_8192": hl.pattern_from_host(*full)}
    sink = torch.empty(lib.hist_ablation_grid(n) * 256, dtype=torch.int32, device="cuda")
    out = torch.empty(256, dtype=torch.int32, device="cuda")
    res = {"bytes": n, "stages": ["read+write", "+init", "+pattern", "+atomics", "+reduce",
                                  "complete, warp-aggregated increments",
                                  "complete, input staged by bulk copies (cp.async.bulk, 2 x 16 KiB per CTA)"]}
    for law_name, law in (("uniform", synth.uniform()), ("normal_sigma8", synth.normal(128, 8))):
        x = torch.empty(n, dtype=torch.uint8, device="cuda")
        synth.device_fill(x.data_ptr(), n, law, synth.SEED_BASE + 13, 0, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        for name, pd in pats.items():
            row = []
            for stage in range(1, 8):
                def step(stage=stage, pd=pd):
                    _abi.check("hist_ablation", lib.hist_ablation(
                        x.data_ptr(), n, pd.data_ptr() if pd is not None else None, stage,
                        out.data_ptr(), sink.data_ptr(), torch.cuda.current_stream().cuda_stream))
                el = time_steps(torch, step, 2, steps)
                row.append(round(n * steps / el / 1e9, 1))
            res["%s_%s_gbs" % (law_name, name)] = row
        del x
    return res


def table2_extras(torch, hl, synth, steps=10, n=1 << 30):
    """Table 2 on this GPU: GB/s of the per-warp kernel and of the adaptive
    kernel (with the 960-slot pattern the rule derives from the input's own
    histogram, and with the full 8192-slot table) on the paper's inputs:
    random (uniform), sequential (x[i] = i mod 256), all 127, all 1 and
    clamp(round(N(128, 8))) for the missing X-ray data.  Each input is 1 GiB
    of that law (the paper's 8192 x 8192 slice would sit in the 129 MB L2)."""
    out = {"bytes": n, "inputs": ["random", "sequential", "all127", "all1", "xray_normal_sigma8"]}
    full = hl.pattern_from_host([32 * b for b in range(256)], [5] * 256, 8192, 8192)
    x = torch.empty(n, dtype=torch.uint8, device="cuda")
    cs = torch.cuda.current_stream().cuda_stream
    o = hl.empty_hist()
    rows = {"plain_gbs": [], "adaptive_960_gbs": [], "adaptive_8192_gbs": []}
    for name in out["inputs"]:
        if name == "sequential":
            synth.device_ramp(x.data_ptr(), n, 0, cs)
        else:
            law = {"random": synth.uniform(), "all127": synth.constant(127), "all1": synth.constant(1),
                   "xray_normal_sigma8": synth.normal(128, 8)}[name]
            synth.device_fill(x.data_ptr(), n, law, synth.SEED_BASE + 17, 0, cs)
        # the rule's 960-slot pattern from the input's own histogram, on the device
        pd = hl.binning_pattern(hl.hist_plain(x, o), 960)
        torch.cuda.synchronize()
        for key, fn in (("plain_gbs", lambda: hl.hist_plain(x, o)),
                        ("adaptive_960_gbs", lambda: hl.hist_adaptive(x, pd, o)),
                        ("adaptive_8192_gbs", lambda: hl.hist_adaptive(x, full, o))):
            el = time_steps(torch, fn, 2, steps)
            rows[key].append(round(n * steps / el / 1e9, 1))
    out.update(rows)
    del x
    return out


def serving_extras(torch, np, hl, synth, hbm, rates=SERVE_RATES):
    """The serving workload: Poisson arrivals over 256 streams with 64 MiB
    payload regions each (16 GiB resident), sizes log-uniform in 4 KiB ..
    64 MiB, 20% of the streams degenerate, a 32 GiB admission budget; the
    schedule is replayed in real time by the library's own loop.  Per rate:
    offered and served GB/s and request latency (completion seen by the host
    - scheduled arrival) percentiles.  `capacity` submits a whole schedule at
    t = 0."""
    from paper_1011_0235_gb300 import _abi
    from synth import workloads

    streams, region = 256, 64 * MiB
    seed = synth.SEED_BASE + 5
    laws = workloads.serving_streams(streams, region, seed=seed)
    pool = torch.empty(streams * region + 16, dtype=torch.uint8, device="cuda")
    cs = torch.cuda.current_stream().cuda_stream
    for law in laws:
        synth.device_fill(pool.data_ptr() + law.offset, region, law.thr, seed, law.counter0, cs)
    torch.cuda.synchronize()
    out = {"streams": streams, "payload_pool_bytes": streams * region, "hbm_budget": 32 << 30}

    def run(reqs, at_zero=False, mode=hl.MODE_AUTO, base=None):
        count = len(reqs)
        base = pool.data_ptr() if base is None else base
        outs = torch.empty((count, 256), dtype=torch.int32, device="cuda")
        R = (_abi.Request * count)()
        for i, r in enumerate(reqs):
            R[i].arrival_ns = 0 if at_zero else r.arrival_ns
            R[i].stream, R[i].d_in, R[i].n = r.stream, base + r.offset, r.n
            R[i].d_out, R[i].tag = outs.data_ptr() + i * 1024, i
        torch.cuda.synchronize()
        srv = hl.Server(streams=streams, mode=mode)
        k = min(count, 64)
        srv.replay((_abi.Request * k)(*R[:k]), timeout_ms=60000)  # warm-up: first launches, clocks
        # and a burst at t = 0, which batches more than 32 requests (the large kernel variant)
        burst = (_abi.Request * k)(*R[:k])
        for i in range(k):
            burst[i].arrival_ns = 0
        srv.replay(burst, timeout_ms=60000)
        srv.close()
        srv = hl.Server(streams=streams, mode=mode)
        done = srv.replay(R, timeout_ms=120000)
        st = srv.stats()
        srv.close()
        c = np.frombuffer(done, dtype=np.uint64).reshape(count, 6)
        lat = (c[:, 5] - c[:, 3]).astype(np.float64) / 1e3  # us
        queued = (c[:, 4] - c[:, 3]).astype(np.float64) / 1e3  # arrival -> batch launched
        on_gpu = (c[:, 5] - c[:, 4]).astype(np.float64) / 1e3  # launched -> completion seen
        nb = float(sum(r.n for r in reqs))
        span = (float(c[:, 5].max()) - (0.0 if at_zero else float(reqs[0].arrival_ns))) / 1e9
        ok = bool(np.array_equal(outs.sum(dim=1, dtype=torch.int64).cpu().numpy(),
                                 np.array([r.n for r in reqs], np.int64)))
        return {"requests": count, "bytes": int(nb), "served_gbs": round(nb / span / 1e9, 2),
                "p50_us": round(float(np.percentile(lat, 50)), 1), "p99_us": round(float(np.percentile(lat, 99)), 1),
                "p999_us": round(float(np.percentile(lat, 99.9)), 1), "max_us": round(float(lat.max()), 1),
                "p50_queued_us": round(float(np.percentile(queued, 50)), 1),
                "p50_launched_to_done_us": round(float(np.percentile(on_gpu, 50)), 1),
                "batches": int(st.batches), "mean_batch": round(count / max(1, st.batches), 2),
                "sums_equal_sizes": ok}

    for lam in rates:
        reqs = workloads.serving_schedule(lam, int(lam * SERVE_SECONDS), streams=streams, region=region,
                                          seed=synth.SEED_BASE + 6 + lam)
        r = run(reqs)
        r["offered_gbs"] = round(sum(q.n for q in reqs) / (reqs[-1].arrival_ns / 1e9) / 1e9, 2)
        out["rate_%d" % lam] = r
    reqs = workloads.serving_schedule(50000, 4000, streams=streams, region=region, seed=synth.SEED_BASE + 7)
    cap = run(reqs, at_zero=True)
    cap["frac_of_hbm"] = round(cap["served_gbs"] / hbm, 4)
    # the counting kernels' own rate on this mix: each stream's 64 MiB region
    # counted once by the kernel AUTO gives its law (one-shot calls on 64 MiB,
    # launch included), the requests' bytes weighted by it
    o = hl.empty_hist()

    def t_of(f):
        f()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(3):
            f()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / 3 / 1e3

    rate = []
    for law in laws:
        x = pool[law.offset:law.offset + region]
        if law.kind == "degenerate":
            p = hl.binning_pattern(hl.hist_plain(x, o).clone(), 8192)
            rate.append(region / t_of(lambda: hl.hist_adaptive(x, p, o)))
        else:
            rate.append(region / t_of(lambda: hl.hist_plain(x, o)))
    nbytes = float(sum(r.n for r in reqs))
    cap["auto_kernels_alone_gbs"] = round(nbytes / sum(r.n / rate[r.stream] for r in reqs) / 1e9, 1)
    out["capacity"] = cap
    # the same burst with every stream in ADAPTIVE mode
    cad = run(reqs, at_zero=True, mode=hl.MODE_ADAPTIVE)
    cad["frac_of_hbm"] = round(cad["served_gbs"] / hbm, 4)
    out["capacity_adaptive"] = cad
    del pool
    # the host-fed variant: the payloads stay in pinned host memory and the
    # batch kernels read them over the host link (a 1 GiB pool of 256 streams
    # with 4 MiB regions; a burst of 2000 requests of 4 KiB .. 4 MiB, AUTO
    # mode), beside the same burst from a device copy of the pool
    hregion = 4 * MiB
    hlaws = workloads.serving_streams(streams, hregion, seed=seed)
    pool = torch.empty(streams * hregion + 16, dtype=torch.uint8, device="cuda")
    for law in hlaws:
        synth.device_fill(pool.data_ptr() + law.offset, hregion, law.thr, seed, law.counter0, cs)
    hpool = torch.empty(pool.numel(), dtype=torch.uint8, pin_memory=True)
    hpool.copy_(pool)
    torch.cuda.synchronize()
    hreqs = workloads.serving_schedule(50000, 2000, streams=streams, region=hregion, size_hi=hregion,
                                       seed=synth.SEED_BASE + 8)
    hf = {"pool_bytes": streams * hregion, "requests": len(hreqs)}
    for name, base in (("pinned_host", hpool.data_ptr()), ("device", pool.data_ptr())):
        r = run(hreqs, at_zero=True, base=base)
        hf[name] = {k: r[k] for k in ("served_gbs", "p50_us", "p99_us", "batches", "sums_equal_sizes")}
    out["capacity_host_fed"] = hf
    del pool, hpool
    return out


# ---------------------------------------------------------- reference ----

def summary_of(ex, value, hbm):
    """The figures the extras are read for, last in the line (a reader of its
    tail sees them): fractions are of the measured HBM copy bandwidth."""
    def g(*path):
        d = ex
        for k in path:
            if not isinstance(d, dict) or k not in d:
                return None
            d = d[k]
        return d
    sm = {"hbm_gbs": hbm, "adaptive_stream_gbs": round(value, 1), "adaptive_frac": round(value / hbm, 4),
          "adaptive_stream_default_gbs": g("adaptive_stream_default_gbs"),
          "plain_stream_gbs": g("plain_stream_gbs"), "plain_stream_default_gbs": g("plain_stream_default_gbs")}
    ad, pl, au = g("degenerate_adaptive_gbs"), g("degenerate_plain_gbs"), g("degenerate_auto_gbs")
    if ad and pl:
        sm["degenerate_gbs"] = {"adaptive": ad, "plain": pl, "auto": au, "auto_window32": g("degenerate_auto_window32_gbs"),
                                "adaptive_over_plain": round(ad / pl, 2),
                                "note": "3x would need %.0f GB/s, above the HBM copy peak: both kernels count in the "
                                        "lane-private table" % (3 * pl)}
    sm["table2_plain_gbs"] = dict(zip(g("table2", "inputs") or [], g("table2", "plain_gbs") or []))
    sm["batch_graph_gbs"] = g("batch_graph_gbs")
    sm["batch_regimes_graph_gbs"] = g("batch_regimes", "graph_gbs")
    cs = g("stream_chunk_sizes")
    if cs:
        sm["chunk_kib"] = cs.get("chunk_kib")
        sm["adaptive_by_chunk_gbs"] = cs.get("adaptive_stream_gbs")
        sm["launch_us_1024x16B"] = cs.get("launch_us_1024x16B")
    sb = g("stream_budgets")
    if sb:
        sm["budgets"] = sb.get("budgets")
        sm["adaptive_by_budget_frac"] = [round(v / hbm, 3) for v in sb.get("adaptive_stream_gbs", [])]
    sv = g("serving")
    if sv:
        sm["serving"] = {k: {"gbs": v.get("served_gbs"), "p50_us": v.get("p50_us"), "p99_us": v.get("p99_us")}
                         for k, v in sv.items() if isinstance(v, dict) and "served_gbs" in v}
        cap = sv.get("capacity") or {}
        if "auto_kernels_alone_gbs" in cap:
            sm["serving"]["capacity"]["auto_kernels_alone_gbs"] = cap["auto_kernels_alone_gbs"]
        hf = sv.get("capacity_host_fed") or {}
        if "pinned_host" in hf:
            sm["serving"]["burst_host_fed_gbs"] = {k: hf[k].get("served_gbs") for k in ("pinned_host", "device")}
    return sm


def run_reference(args):
    world, rank, local = dist_env()
    if rank != 0:
        return 0
    import numpy as np

    import oracle
    import synth

    oracle.build()
    synth.build_host()
    thr = synth.normal(128, 8)
    sample_chunks = 4  # 64 MiB of the workload per step
    chunks = [synth.host(CHUNK, thr, synth.SEED_BASE + 2, c * CHUNK, threads=os.cpu_count() or 1)
              for c in range(sample_chunks)]
    so = oracle.StreamOracle(8192, mode=oracle.MODE_ADAPTIVE)

    def step():
        for ch in chunks:
            so.push(ch)

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        step()
    el = time.perf_counter() - t0
    nbytes = sample_chunks * CHUNK * args.steps
    val = nbytes / el / 1e9
    cfg = workload_config(args.chunks)
    out = {
        "impl": "reference", "metric": METRIC, "value": round(val, 4), "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(el / args.steps * 1e3, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u8", "data": "synthetic",
        "config": cfg,
        "cpu_baseline": {"value": round(val, 4), "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": "%d of the workload's 16 MiB chunks (%d MiB) per step, single-threaded plain C "
                                   "counting loop + degeneracy + binning pattern per chunk"
                                   % (sample_chunks, sample_chunks * 16)},
        "e2e": {"value": round(val, 4), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(out))
    return 0


# -------------------------------------------------------------- native ----

def run_part(args):
    """One workload other than the headline stream, once, for profiling."""
    import numpy as np
    import torch

    import synth
    import paper_1011_0235_gb300 as hl
    from paper_1011_0235_gb300 import build as hbuild

    hbuild.build()
    synth.build()
    hl.lib()
    if args.profile_part == "serving":
        out = serving_extras(torch, np, hl, synth, 6800.0, rates=())
    elif args.profile_part == "ablation":
        out = ablation_extras(torch, hl, synth, 6800.0, steps=1, n=256 << 20)
    elif args.profile_part == "table2":
        out = table2_extras(torch, hl, synth, steps=1, n=256 << 20)
    elif args.profile_part == "auto":
        # the degenerate workload (95 % = 90, switching to uniform every 8
        # chunks) through an AUTO stream: 3 pushes of 64 chunks
        xdg = gen_workload_device(torch, synth, 64, synth.SEED_BASE + 3,
                                  lambda c: synth.degenerate(90, 0.95) if (c // 8) % 2 == 0 else synth.uniform())
        ptrs = [xdg.data_ptr() + c * CHUNK for c in range(64)]
        out = {}
        # a window of one chunk, then a window of 32 chunks (its window
        # kernel), both with the chunks declared complete
        for name, window in (("auto", 1), ("auto_window32", 32)):
            st = hl.Stream(budget=8192, mode=hl.MODE_AUTO, window=window, overlap=True)
            el = time_steps(torch, lambda: st.push_many(ptrs, [CHUNK] * 64), 1, 2)
            out[name + "_gbs"] = round(64 * CHUNK * 2 / el / 1e9, 1)
            out[name + "_recounted"] = st.state().recounted
            st.close()
    elif args.profile_part == "smallchunks":
        # 256 MiB of N(128, 8) in 4096 chunks of 64 KiB through an adaptive
        # stream: one push_many, four counting launches of 1024 chunks
        x = gen_workload_device(torch, synth, 16, synth.SEED_BASE + 2, lambda c: synth.normal(128, 8))
        k, c64 = 4096, 64 << 10
        st = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE)
        cp = x.data_ptr() + np.arange(k, dtype=np.uint64) * np.uint64(c64)
        el = time_steps(torch, lambda: st.push_many(cp, np.full(k, c64, dtype=np.uint64)), 1, 2)
        out = {"smallchunks_gbs": round(k * c64 * 2 / el / 1e9, 1)}
    elif args.profile_part == "budgets":
        # 256 MiB of N(128, 8) counted once by hist_adaptive with the rule's
        # pattern at 960, 2048 and 4096 slots, and once at the full table
        x = gen_workload_device(torch, synth, 16, synth.SEED_BASE + 2, lambda c: synth.normal(128, 8))
        o = hl.empty_hist()
        h = hl.hist_plain(x, o).clone()
        out = {}
        for b in (960, 2048, 4096, 8192):
            pb = hl.binning_pattern(h, b)
            el = time_steps(torch, lambda: hl.hist_adaptive(x, pb, o), 1, 1)
            out["adaptive_%d_gbs" % b] = round(16 * CHUNK / el / 1e9, 1)
    elif args.profile_part == "regimes":
        # the 4096-image batch tuned per regime, then one graph launch
        out = batch_extras(torch, hl, synth, 6800.0, steps=1, autotune=True)
    elif args.profile_part == "budget960":
        # the headline's N(128, 8) stream with the paper's 960-slot pattern:
        # 3 pushes of 64 chunks
        x = gen_workload_device(torch, synth, 64, synth.SEED_BASE + 2, lambda c: synth.normal(128, 8))
        st = hl.Stream(budget=960, mode=hl.MODE_ADAPTIVE)
        ptrs = [x.data_ptr() + c * CHUNK for c in range(64)]
        el = time_steps(torch, lambda: st.push_many(ptrs, [CHUNK] * 64), 1, 2)
        out = {"adaptive_960_gbs": round(64 * CHUNK * 2 / el / 1e9, 1), "status": st.state().status}
    else:
        out = batch_extras(torch, hl, synth, 6800.0, steps=1, autotune=False)
    print(json.dumps({"profile_part": args.profile_part, "result": out}))
    return 0


def run_native(args):
    import numpy as np
    import torch

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    barrier = None
    dist = None
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
        barrier = dist.barrier

    import synth
    import paper_1011_0235_gb300 as hl
    from paper_1011_0235_gb300 import build as hbuild

    hbuild.build()
    synth.build()
    hl.lib()

    chunks = args.chunks
    nbytes = chunks * CHUNK
    thr = synth.normal(128, 8)
    seed = synth.SEED_BASE + 2
    x = gen_workload_device(torch, synth, chunks, seed, lambda c: thr, first_chunk=rank * chunks)
    # chunk tables as arrays, passed to the library without conversion
    ptrs = np.array([x.data_ptr() + c * CHUNK for c in range(chunks)], dtype=np.uint64)
    sizes = np.full(chunks, CHUNK, dtype=np.uint64)

    def stream_step(st):
        def step():
            st.push_many(ptrs, sizes)
            st.flush()
        return step

    st_ad = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE, overlap=True)
    sampler = ClockSampler(local)
    step = stream_step(st_ad)
    if not args.profile:
        sampler.start()
        # settle clocks for at least one second before the timed region
        t_settle = time.time()
        while time.time() - t_settle < 1.0:
            step()
            torch.cuda.synchronize()
    el = time_steps(torch, step, args.warmup, args.steps, barrier)
    clocks = sampler.stop()
    from paper_1011_0235_gb300 import shard
    el = shard.slowest(el, device="cuda")
    value = world * nbytes * args.steps / el / 1e9
    # the adaptive stream at the full table runs batch_flat_kernel: one launch per
    # push_many of up to STREAM_MAX_BATCH chunks, nothing left for flush
    launches_per_step = -(-chunks // STREAM_MAX_BATCH)

    extras = {}
    peaks = measured_peaks()
    hbm = peaks.get("hbm_gbs") if peaks else None
    peak_src = "measured" if hbm else "fallback"
    hbm = hbm or 6800.0

    # dominant (only) kernel of the step: batch_flat_kernel, all chunks
    # of a push_many in one launch; algorithmic bytes = the pixels it reads
    avg_launch_s = el / (args.steps * launches_per_step)
    bytes_per_launch = nbytes // launches_per_step
    achieved = bytes_per_launch / avg_launch_s / 1e9
    roofline = {"bound": "hbm", "achieved": round(achieved, 2), "peak": hbm, "unit": "GB/s",
                "frac": round(achieved / hbm, 4), "traffic": recorded_traffic("batch_flat_kernel"),
                "kernel": "batch_flat_kernel", "peak_source": peak_src,
                "algorithmic_bytes_per_launch": bytes_per_launch,
                "launch_ms": round(avg_launch_s * 1e3, 4)}

    if not args.profile:
        # plain kernel on the same stream of data
        st_pl = hl.Stream(budget=8192, mode=hl.MODE_PLAIN, overlap=True)
        el_pl = time_steps(torch, stream_step(st_pl), args.warmup, args.steps, barrier)
        extras["plain_stream_gbs"] = round(world * nbytes * args.steps / el_pl / 1e9, 2)
        extras["adaptive_stream_gbs"] = round(value, 2)
        extras["adaptive_frac_of_hbm"] = round(value / world / hbm, 4)
        extras["plain_frac_of_hbm"] = round(extras["plain_stream_gbs"] / world / hbm, 4)
        # the same streams without HIST_OVERLAP_PUSHES (the library's default:
        # each launch reads its chunks only after the work before it completes)
        for name, mode in (("adaptive", hl.MODE_ADAPTIVE), ("plain", hl.MODE_PLAIN)):
            sd = hl.Stream(budget=8192, mode=mode)
            eld = time_steps(torch, stream_step(sd), args.warmup, args.steps, barrier)
            extras["%s_stream_default_gbs" % name] = round(world * nbytes * args.steps / eld / 1e9, 2)
            sd.close()
        # degenerate workload: 95 % = 90 + 5 % uniform, switching to uniform every 8 chunks
        xdg = gen_workload_device(torch, synth, chunks, synth.SEED_BASE + 3,
                                  lambda c: synth.degenerate(90, 0.95) if (c // 8) % 2 == 0 else synth.uniform())
        pd = [xdg.data_ptr() + c * CHUNK for c in range(chunks)]
        for name, mode, window in (("auto", hl.MODE_AUTO, 1), ("plain", hl.MODE_PLAIN, 1),
                                   ("adaptive", hl.MODE_ADAPTIVE, 1), ("auto_window32", hl.MODE_AUTO, 32)):
            s2 = hl.Stream(budget=8192, mode=mode, window=window, overlap=True)

            def st2(s2=s2):
                s2.push_many(pd, sizes)
                s2.flush()
            e2 = time_steps(torch, st2, args.warmup, args.steps, barrier)
            extras["degenerate_%s_gbs" % name] = round(world * nbytes * args.steps / e2 / 1e9, 2)
            s2.close()
        # the adaptive stream below the full table on the same data
        row = []
        for b in (960, 2048, 4096):
            s3 = hl.Stream(budget=b, mode=hl.MODE_ADAPTIVE)

            def st3(s3=s3):
                s3.push_many(pd, sizes)
            e5 = time_steps(torch, st3, 2, 10)
            row.append(round(nbytes * 10 / e5 / 1e9, 2))
            s3.close()
        extras["stream_budgets_degenerate"] = {"budgets": [960, 2048, 4096], "adaptive_stream_gbs": row,
                                               "frac_of_hbm": [round(v / hbm, 4) for v in row]}
        del xdg
        extras.update(batch_extras(torch, hl, synth, hbm, steps=max(3, min(args.steps, 10))))
        extras["serving"] = serving_extras(torch, np, hl, synth, hbm)
        extras["ablation_table1"] = ablation_extras(torch, hl, synth, hbm)
        # a read-only kernel's ceiling on this GPU: stage 1 reads every 16-byte
        # vector once and writes 1 KiB per CTA (the copy peak reads and writes)
        abl = extras["ablation_table1"]
        extras["read_only_kernel_gbs"] = max(abl[k][0] for k in abl if k.endswith("_gbs"))
        extras["table2"] = table2_extras(torch, hl, synth)
        # one-shot kernels on the whole 1 GiB at once (no stream)
        full = hl.pattern_from_host([32 * b for b in range(256)], [5] * 256, 8192, 8192)
        o = hl.empty_hist()
        e3 = time_steps(torch, lambda: hl.hist_adaptive(x, full, o), 2, 10)
        extras["oneshot_adaptive_full_table_gbs"] = round(nbytes * 10 / e3 / 1e9, 2)
        e4 = time_steps(torch, lambda: hl.hist_plain(x, o), 2, 10)
        extras["oneshot_plain_gbs"] = round(nbytes * 10 / e4 / 1e9, 2)
        st_pl.close()
        # the same stream below the full table (the paper's 960 slots and
        # between); beside it, one hist_adaptive call over the same bytes with
        # the rule's pattern
        sb = {"budgets": [960, 2048, 4096]}
        hx1 = hl.hist_plain(x, hl.empty_hist())
        for name, mode in (("adaptive", hl.MODE_ADAPTIVE), ("auto", hl.MODE_AUTO)):
            row = []
            for b in sb["budgets"]:
                s3 = hl.Stream(budget=b, mode=mode)

                def st3(s3=s3):
                    s3.push_many(ptrs, sizes)
                    s3.flush()
                e5 = time_steps(torch, st3, 2, 10)
                row.append(round(nbytes * 10 / e5 / 1e9, 2))
                s3.close()
            sb["%s_stream_gbs" % name] = row
        row = []
        for b in sb["budgets"]:
            pb = hl.binning_pattern(hx1.clone(), b)
            e6 = time_steps(torch, lambda: hl.hist_adaptive(x, pb, o), 2, 10)
            row.append(round(nbytes * 10 / e6 / 1e9, 2))
        sb["oneshot_adaptive_gbs"] = row
        sb["adaptive_frac_of_hbm"] = [round(v / hbm, 4) for v in sb["adaptive_stream_gbs"]]
        extras["stream_budgets"] = sb
        # the same 1 GiB pushed as smaller chunks (one push_many per GiB):
        # the fixed cost per launch and per chunk against the bytes
        cs = {"chunk_kib": [16384, 1024, 256, 64]}
        for name, mode in (("adaptive", hl.MODE_ADAPTIVE), ("auto", hl.MODE_AUTO)):
            row = []
            for kib in cs["chunk_kib"]:
                k = nbytes // (kib << 10)
                cp = x.data_ptr() + np.arange(k, dtype=np.uint64) * np.uint64(kib << 10)
                cz = np.full(k, kib << 10, dtype=np.uint64)
                s4 = hl.Stream(budget=8192, mode=mode, overlap=True)

                def st4(s4=s4, cp=cp, cz=cz):
                    s4.push_many(cp, cz)
                e7 = time_steps(torch, st4, 2, 5)
                row.append(round(nbytes * 5 / e7 / 1e9, 2))
                s4.close()
            cs["%s_stream_gbs" % name] = row
            # the fixed cost: one launch of 1024 chunks of 16 bytes
            tp = x.data_ptr() + np.arange(1024, dtype=np.uint64) * np.uint64(4096)
            tz = np.full(1024, 16, dtype=np.uint64)
            s5 = hl.Stream(budget=8192, mode=mode, overlap=True)
            e8 = time_steps(torch, lambda: s5.push_many(tp, tz), 3, 20)
            cs.setdefault("launch_us_1024x16B", {})[name] = round(e8 / 20 * 1e6, 1)
            s5.close()
        extras["stream_chunk_sizes"] = cs

    # end to end: host buffers through hist_stream_push_host, H2D inside the timed region
    e2e = None
    try:
        if args.profile:
            raise RuntimeError("skipped (--profile)")
        hx = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
        synth._host_lib().synth_fill_host_mt(hx.data_ptr(), nbytes, np.ascontiguousarray(thr).ctypes.data,
                                             seed, 0, os.cpu_count() or 1)
        st_e = hl.Stream(budget=8192, mode=hl.MODE_ADAPTIVE)
        st_e.attach_staging(CHUNK, 3)
        tot_d = torch.empty(256, dtype=torch.int64, device="cuda")
        tot_h = torch.empty(256, dtype=torch.int64, pin_memory=True)

        def e2e_step():
            for c in range(chunks):
                st_e.push_host(hx.data_ptr() + c * CHUNK, CHUNK)
            st_e.totals(tot_d)
            tot_h.copy_(tot_d, non_blocking=True)

        ksteps = max(3, min(args.steps, 20))
        # three timed windows of ksteps steps each, the median reported: the
        # host thread enqueues a copy and a launch per chunk, and a stall of
        # it in one window (tens of ms were seen on the shared host) would
        # otherwise decide the figure
        wins = [time_steps(torch, e2e_step, w, ksteps, barrier) for w in (max(args.warmup, 3), 1, 1)]
        el_e = shard.slowest(sorted(wins)[1], device="cuda")
        # the link's own ceiling: a plain 1 GiB pinned-host -> device copy
        # (the median of three windows of three copies)
        dx = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        el_c = sorted(time_steps(torch, lambda: dx.copy_(hx, non_blocking=True), 1, 3) for _ in range(3))[1]
        del dx
        e2e = {"value": round(world * nbytes * ksteps / el_e / 1e9, 2), "unit": UNIT,
               "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": 256 * 8, "steps": ksteps,
               "windows_gbs": [round(world * nbytes * ksteps / w / 1e9, 2) for w in wins],
               "path": "hist_stream_push_host: pinned host memory read by the counting kernels over the host link, a "
                       "chunk's reads beside the launch before; median of three windows of `steps` steps",
               "h2d_copy_gbs": round(nbytes * 3 / el_c / 1e9, 2)}
        st_e.close()
        if world == 1:
            extras["host_fed"] = host_fed_extras(torch, hl, hx, chunks, 5)
            extras["host_fed"]["h2d_copy_gbs"] = e2e["h2d_copy_gbs"]
        del hx
    except Exception as exc:  # report, do not hide
        e2e = {"value": None, "unit": UNIT, "error": repr(exc)}

    cpu = None
    if rank == 0 and world == 1 and not args.profile:
        import oracle

        oracle.build()
        sample = 8
        host_chunks = [synth.host(CHUNK, thr, seed, c * CHUNK, threads=os.cpu_count() or 1) for c in range(sample)]
        rate, done, secs = cpu_oracle_rate(host_chunks, CPU_SAMPLE_SECONDS)
        cpu = {"value": round(rate, 4), "unit": UNIT, "cores": 1, "kind": "oracle",
               "sample": "the first %d chunks (%d MiB) of the workload, repeated for %.1f s (%d MiB processed); "
                         "single-threaded C counting loop + degeneracy + binning pattern per chunk"
                         % (sample, sample * 16, secs, done // MiB)}
        # the oracle's counting loop on every host core (its own slice and
        # histogram per thread, summed): a second, parallel CPU reference point
        threads = os.cpu_count() or 1
        hbuf = np.concatenate(host_chunks)
        trate, tdone, tsecs, thist = cpu_oracle_threads_rate(hbuf, CPU_THREADS_SECONDS, threads)
        if not np.array_equal(thist, oracle.hist(hbuf)):
            raise RuntimeError("threaded oracle count differs from the oracle")
        extras["cpu_oracle_threads"] = {
            "value": round(trate, 3), "unit": UNIT, "cores": threads, "kind": "oracle counting loop per thread",
            "sample": "the first %d chunks (%d MiB), split into %d contiguous slices, repeated for %.1f s (%d MiB)"
                      % (sample, sample * 16, threads, tsecs, tdone // MiB)}

    if extras and not args.profile:
        extras["summary"] = summary_of(extras, value, hbm)

    if rank == 0:
        out = {
            "metric": METRIC, "value": round(value, 2), "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(el / args.steps * 1e3, 4), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u8", "data": "synthetic",
            "config": workload_config(chunks), "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e,
            "clocks": clocks, "gpu_launches": launches_per_step * args.steps, "extras": extras,
        }
        print(json.dumps(out))
    st_ad.close()
    if world > 1:
        dist.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.profile_part:
        return run_part(args)
    return run_native(args)


if __name__ == "__main__":
    sys.exit(main())
