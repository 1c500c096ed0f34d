#!/usr/bin/env python
"""Benchmark of the GB300 Hamming decoder.

Default workload (one "step"): the single-n sweep -- Hamming (15,11), (31,26)
and (63,57), 2^24 codewords each, packed LSB-first uint32 streams of encoded
uniform data with single-bit errors (p1 = 0.1) and double-bit errors
(p2 = 0.01), u8 syndromes and an error count.  A step decodes all three
streams (one hd_decode call each).  Inputs are resident in HBM before the
timed region; the three streams and their outputs (475 MB) are larger than
L2 and each buffer is touched once per step.

Prints ONE JSON line (rank 0) on stdout: the step's figures and one or two of each
section; the sections in full go to stderr as a JSON line of their own, so that
the line stays short enough for readers that keep only the end of the output.
``--impl reference`` times the CPU oracle on
the host cores instead (the reference arm of this workload).
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

SWEEP_CODES = (15, 31, 63)
SWEEP_N = 1 << 24
SWEEP_P1, SWEEP_P2 = 0.1, 0.01
ROOFLINE_N = 63  # the dominant kernel of a sweep step (largest byte count)
METRIC = "decoded Gbit/s"
WORKLOAD = ("single-n sweep: Hamming (15,11), (31,26), (63,57); 2^24 codewords each; packed LSB-first "
            "uint32 streams; encoded uniform data (seed n), single-bit error p1=0.1 and double-bit p2=0.01 "
            "per codeword; u8 syndromes + err_count")


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--e2e-steps", type=int, default=30)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0, help="target CPU time of the oracle baseline")
    ap.add_argument("--codes", type=str, default=",".join(map(str, SWEEP_CODES)),
                    help="subset of the sweep codes to run (profiling a single kernel)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-adt", action="store_true", help="skip the SDT vs ADT (Eq. 1) transfer section")
    ap.add_argument("--no-autotune", action="store_true",
                    help="keep the built-in kernel configurations (the sweep autotunes each code by default)")
    ap.add_argument("--pin", type=str, default="",
                    help="n:i,... pin configuration i of code n (u8 syndromes) instead of autotuning it (for ncu)")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched mixed-n section")
    ap.add_argument("--batched-only", action="store_true", help="run only the batched mixed-n section")
    ap.add_argument("--batched-packets", type=int, default=10000)
    ap.add_argument("--batched-steps", type=int, default=20)
    ap.add_argument("--batched-config", type=int, default=-1,
                    help="pin batch-kernel configuration I instead of hd_plan_autotune (e.g. for ncu)")
    ap.add_argument("--no-serve", action="store_true", help="skip the serving section")
    ap.add_argument("--serve-only", action="store_true", help="run only the serving section")
    ap.add_argument("--serve-packets", type=int, default=100000)
    ap.add_argument("--serve-rates", type=str, default="1e4,1e5,1e6", help="Poisson arrival rates, packets/s")
    ap.add_argument("--serve-saturation-rates", type=str, default="2e6,4e6,8e6",
                    help="higher rates tried in order until the server saturates")
    ap.add_argument("--no-serve-host", action="store_true", help="skip serving from pinned host memory")
    ap.add_argument("--no-shortened", action="store_true", help="skip the shortened-code (M, t) grid section")
    ap.add_argument("--shortened-only", action="store_true", help="run only the shortened-code section")
    ap.add_argument("--short-steps", type=int, default=10, help="timed launches per (M, t) configuration")
    ap.add_argument("--short-grid", type=str, default="", help="subset of the (M, t) grid, e.g. 2000:2,400:6")
    ap.add_argument("--short-no-autotune", action="store_true", help="keep the built-in tile configuration")
    ap.add_argument("--no-secded", action="store_true", help="skip the SECDED section")
    ap.add_argument("--secded-only", action="store_true", help="run only the SECDED section")
    ap.add_argument("--secded-codes", type=str, default="15,31,63,127,255")
    ap.add_argument("--no-per-code", action="store_true", help="skip the per-code section (configs 1-3, p1 grid)")
    ap.add_argument("--per-code-only", action="store_true", help="run only the per-code section")
    ap.add_argument("--per-code-codes", type=str, default="", help="subset of the per-code section's codes")
    return ap.parse_args()


def code_params(n):
    m = (n + 1).bit_length() - 1
    return m, n - m


def algorithmic_bytes(n, N, syn_bytes=1):
    """Bytes one decode must move: n/8 read + k/8 written + syndromes per codeword."""
    m, k = code_params(n)
    return (N * n + 7) // 8 + (N * k + 7) // 8 + N * syn_bytes


def dist_setup(gpus):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world != gpus:
        if world == 1 and gpus > 1:
            raise SystemExit("--gpus N > 1 must be launched with torch.distributed.run (one rank per GPU)")
    return rank, world, local


# The sources the roofline kernel (the n = 63 streaming decoder) is compiled from.
ROOFLINE_SOURCES = ("hd_device.cuh", "hd_tile.cuh", "hd_stream.cuh", "hd_stream_b.cu")


def kernel_sources_hash():
    """sha256 over the roofline kernel's sources (names and contents)."""
    import hashlib
    pkg = os.path.join(ROOT, "paper_1412_6862_gb300", "csrc")
    files = [os.path.join(pkg, f) for f in ROOFLINE_SOURCES]
    h = hashlib.sha256()
    for f in files:
        h.update(os.path.basename(f).encode())
        with open(f, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def recorded_traffic(kernel_desc):
    """DRAM bytes per launch of the roofline kernel from the committed ncu records
    (one per configuration the autotuner may choose), or None when no record is
    for this configuration or the kernel sources changed since it was taken."""
    p = os.path.join(ROOT, "profiles", "roofline_traffic_n63.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        recs = json.load(f).get("records", [])
    h = kernel_sources_hash()
    for rec in recs:
        if rec.get("sources_sha256") == h and rec.get("kernel") == kernel_desc:
            return int(rec["dram_bytes_read"]) + int(rec["dram_bytes_write"])
    return None


def reduce_max(value, device=None):
    """Max of a float over all ranks (the value itself when not distributed)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(value)
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def weak_scaling_value(units_per_rank, world, seconds):
    """Whole-job throughput: the units all ranks processed over the slowest rank's time."""
    return units_per_rank * world / seconds


def shard_seed(n, rank):
    """Every rank decodes its own shard: the same workload with rank-specific data."""
    return n + 1000 * rank


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi clock/throttle sampling during the timed region."""

    FIELDS = ("uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid: str | None, interval_ms: int = 20):
        self.uuid = (uuid or "").lower().replace("gpu-", "").replace("-", "")
        self.tmp = tempfile.NamedTemporaryFile(prefix="hdclk", suffix=".csv", delete=False)
        self.proc = None
        self.interval_ms = interval_ms

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", str(self.interval_ms)], stdout=self.tmp, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        time.sleep(0.15)
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        self.tmp.close()

    def summary(self):
        rows = []
        try:
            with open(self.tmp.name) as f:
                for line in f:
                    parts = [x.strip() for x in line.split(",")]
                    if len(parts) < 9:
                        continue
                    u = parts[0].lower().replace("gpu-", "").replace("-", "")
                    if self.uuid and u != self.uuid:
                        continue
                    rows.append(parts)
        finally:
            os.unlink(self.tmp.name)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        # samples under load: the upper half of the SM clock distribution
        sm_sorted = sorted(sm)
        return {"sm_mhz": float(np.median(sm_sorted[len(sm_sorted) // 2:])) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------------------
# CPU oracle timing (baseline and reference arm)
# ---------------------------------------------------------------------------
def oracle_sample_inputs(codes, per_code):
    import oracle
    from paper_1412_6862_gb300 import synth
    out = {}
    for n in codes:
        m, k = code_params(n)
        N = per_code[n]
        data = synth.random_words(n, N * k)
        s = oracle.encode(data, n, N)
        synth.apply_errors(s, synth.error_events(n, n, N, p1=SWEEP_P1, p2=SWEEP_P2))
        out[n] = s
    return out


def oracle_decode_all(streams, per_code, threads):
    import oracle
    bits = 0
    for n, s in streams.items():
        m, k = code_params(n)
        N = per_code[n]
        outb = np.zeros((N * k + 31) // 32, np.uint32)
        syn = np.zeros(N, np.uint8)
        oracle.decode_threaded(s, n, N, oracle.SYN_U8, threads, outb, syn)
        bits += N * k
    return bits


def calibrate_oracle(threads, seconds):
    """Codewords per code so that one pass over the three codes takes ~seconds."""
    probe = {n: 1 << 15 for n in SWEEP_CODES}
    streams = oracle_sample_inputs(SWEEP_CODES, probe)
    t0 = time.perf_counter()
    oracle_decode_all(streams, probe, threads)
    dt = max(time.perf_counter() - t0, 1e-3)
    scale = seconds / dt
    return {n: int(max(1 << 12, min(SWEEP_N, (probe[n] * scale) // 32 * 32))) for n in SWEEP_CODES}


def cpu_baseline(seconds):
    threads = os.cpu_count() or 1
    per_code = calibrate_oracle(threads, seconds)
    streams = oracle_sample_inputs(SWEEP_CODES, per_code)
    t0 = time.perf_counter()
    bits, passes = 0, 0
    while True:
        bits += oracle_decode_all(streams, per_code, threads)
        passes += 1
        if time.perf_counter() - t0 >= seconds:
            break
    dt = time.perf_counter() - t0
    return {"value": bits / dt / 1e9, "unit": "Gbit/s", "cores": threads, "kind": "oracle",
            "sample": f"{passes} pass(es) over the first {per_code[15]}/{per_code[31]}/{per_code[63]} codewords of the "
                      f"(15,11)/(31,26)/(63,57) streams, bit-by-bit C oracle on {threads} host threads, {dt:.1f} s"}


def run_reference(args):
    rank, world, local = dist_setup(args.gpus)
    if rank != 0:
        return
    threads = os.cpu_count() or 1
    # a step decodes a bounded sample of each stream; the whole run stays within minutes
    budget = min(6.0, 150.0 / max(1, args.steps + args.warmup))
    per_code = calibrate_oracle(threads, budget)
    streams = oracle_sample_inputs(SWEEP_CODES, per_code)
    for _ in range(args.warmup):
        oracle_decode_all(streams, per_code, threads)
    t0 = time.perf_counter()
    bits = 0
    for _ in range(args.steps):
        bits += oracle_decode_all(streams, per_code, threads)
    dt = time.perf_counter() - t0
    value = bits / dt / 1e9
    line = {"metric": METRIC, "value": value, "unit": "Gbit/s", "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": dt / max(1, args.steps) * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOAD, "sample_codewords": per_code},
            "cpu_baseline": {"value": value, "unit": "Gbit/s", "cores": threads, "kind": "oracle",
                             "sample": f"{per_code} codewords per stream per step, bit-by-bit C oracle"},
            "e2e": {"value": value, "unit": "Gbit/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# Batched mixed-n workload
# ---------------------------------------------------------------------------
BATCH_P1 = 0.05


def align4(w):
    return (w + 3) // 4 * 4


def build_batched(dev, num_packets, seed=0, lengths=None):
    """The batched configuration: packets with n uniform over the six codes (or
    over ``lengths``) and log-uniform lengths, every buffer 16-byte aligned
    inside three arenas.  Codewords come from the GPU encoder; channel errors
    from the generator."""
    import torch
    from paper_1412_6862_gb300 import hd, synth
    specs = synth.packet_table(seed, num_packets) if lengths is None else \
        synth.packet_table(seed, num_packets, lengths=tuple(lengths))
    layout = []
    tin = tout = tsyn = tdat = 0
    for sp in specs:
        m, k = code_params(sp.n)
        iw, ow, dw = hd.words_for(sp.num_codewords * sp.n), hd.words_for(sp.num_codewords * k), \
            hd.words_for(sp.num_codewords * k)
        layout.append((sp.n, sp.num_codewords, tin, tout, tsyn, tdat, iw, ow, dw))
        tin += align4(iw)
        tout += align4(ow)
        tsyn += (sp.num_codewords + 15) // 16 * 16
        tdat += align4(dw)
    data_h = np.zeros(tdat, np.uint32)
    for j, (n, N, oi, oo, osy, od, iw, ow, dw) in enumerate(layout):
        m, k = code_params(n)
        data_h[od:od + dw] = synth.random_words(seed * 100003 + j, N * k)
    d_data = torch.from_numpy(data_h.view(np.int32)).to(dev)
    d_in = torch.zeros(tin, dtype=torch.int32, device=dev)
    base_in, base_data = d_in.data_ptr(), d_data.data_ptr()
    sh = torch.cuda.current_stream(dev).cuda_stream
    for (n, N, oi, oo, osy, od, iw, ow, dw) in layout:
        hd.check(hd.hd_encode(base_data + 4 * od, n, N, base_in + 4 * oi, sh), "hd_encode")
    # channel errors: flip bits on the device, one XOR per touched word
    words, masks = [], []
    for j, (n, N, oi, oo, osy, od, iw, ow, dw) in enumerate(layout):
        b = synth.error_events(seed * 100003 + j, n, N, p1=BATCH_P1).stream_bits()
        words.append(oi + (b >> 5))
        masks.append((np.uint32(1) << (b & 31).astype(np.uint32)))
    wv = np.concatenate(words)
    mv = np.concatenate(masks)
    order = np.argsort(wv, kind="stable")
    wv, mv = wv[order], mv[order]
    uniq, start = np.unique(wv, return_index=True)
    mx = np.bitwise_xor.reduceat(mv, start) if wv.size else mv
    idx = torch.from_numpy(uniq.astype(np.int64)).to(dev)
    msk = torch.from_numpy(mx.view(np.int32)).to(dev)
    d_in[idx] = torch.bitwise_xor(d_in[idx], msk)
    del d_data
    d_out = torch.empty(max(1, tout), dtype=torch.int32, device=dev)
    d_syn = torch.empty(max(16, tsyn), dtype=torch.uint8, device=dev)
    torch.cuda.synchronize(dev)
    return layout, d_in, d_out, d_syn


def run_batched(dev, args, peak, keep_pool=False):
    import torch
    from paper_1412_6862_gb300 import hd
    t_setup = time.perf_counter()
    layout, d_in, d_out, d_syn = build_batched(dev, args.batched_packets)
    P = len(layout)
    bi, bo, bs = d_in.data_ptr(), d_out.data_ptr(), d_syn.data_ptr()
    rows = [(bi + 4 * oi, bo + 4 * oo, bs + osy, N, n, hd.SYN_U8) for (n, N, oi, oo, osy, od, iw, ow, dw) in layout]
    table = hd.packet_table(rows)
    err = torch.empty(P, dtype=torch.int64, device=dev)
    bits = sum(N * code_params(n)[1] for (n, N, *_r) in layout)
    nbytes = sum((N * n + 7) // 8 + (N * code_params(n)[1] + 7) // 8 + N for (n, N, *_r) in layout)
    stream = torch.cuda.current_stream(dev)
    sh = stream.cuda_stream
    plan = hd.hd_plan_create(table, P)
    if args.batched_config >= 0:
        hd.hd_plan_select(plan, args.batched_config)
        tuned = hd.hd_plan_get_info(plan)
    else:
        tuned = hd.hd_plan_autotune(plan, 2, stream)
    setup_s = time.perf_counter() - t_setup

    def timed(fn, reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        fn()
        torch.cuda.synchronize(dev)
        a.record(stream)
        for _ in range(reps):
            fn()
        b.record(stream)
        torch.cuda.synchronize(dev)
        return a.elapsed_time(b) / 1e3 / reps

    def persistent():
        hd.check(hd.hd_plan_launch(plan, err.data_ptr(), sh), "hd_plan_launch")

    t_pers = timed(persistent, args.batched_steps)

    def per_packet(cuda_stream):
        for (a, b, c, N, n, st) in rows:
            rc = hd.hd_decode(a, N * n, n, N, b, c, st, None, cuda_stream)
            if rc != 0:
                raise hd.HDError(rc, "hd_decode")

    t_eager = timed(lambda: per_packet(sh), 2)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        per_packet(torch.cuda.current_stream(dev).cuda_stream)
    t_graph = timed(g.replay, 3)
    del g
    hd.hd_plan_destroy(plan)
    gbps = lambda t: bits / t / 1e9
    res = {
        "workload": f"batched mixed-n: {P} packets, n uniform over {{7,15,31,63,127,255}}, length log-uniform "
                    f"64 bit..4 Mbit rounded to whole codewords, p1={BATCH_P1}, u8 syndromes + per-packet err_count",
        "packets": P, "codewords": int(sum(N for (n, N, *_r) in layout)), "decoded_bits": int(bits),
        "algorithmic_bytes": int(nbytes),
        "persistent_graph": {"gbps": gbps(t_pers), "ms": t_pers * 1e3, "hbm_frac": nbytes / t_pers / 1e9 / peak,
                             "variant": tuned["variant"], "num_variants": tuned["num_variants"],
                             "warps_per_cta": tuned["warps_per_cta"], "stages": tuned["stages"],
                             "tiles": tuned["num_tiles"]},
        "per_packet_eager": {"gbps": gbps(t_eager), "ms": t_eager * 1e3},
        "per_packet_graph": {"gbps": gbps(t_graph), "ms": t_graph * 1e3},
        "speedup_vs_per_packet_eager": t_eager / t_pers,
        "speedup_vs_per_packet_graph": t_graph / t_pers,
        "setup_s": setup_s,
    }
    if keep_pool:
        return res, (layout, d_in, d_out, d_syn)
    return res


# The paper's evaluation grid (Sec. IV-A): packets of M bytes cut into t
# segments, each a shortened Hamming codeword (hd_segment_params).
SHORT_GRID = [(M, t) for M in (400, 800, 1200, 1600, 2000) for t in (2, 3, 4, 5, 6)]
SHORT_INPUT_BYTES = 256 << 20  # per configuration: larger than L2, so every launch streams from HBM
SHORT_P1, SHORT_P2 = 0.05, 0.005


def run_shortened(dev, args, peak):
    """Decode throughput over the paper's (M, t) grid: for each configuration
    ~256 MB of packets, all t segments of all packets in one hd_decode_short
    launch (u16 syndromes, both counters), after hd_short_autotune for that
    segment length.  The bit-by-bit oracle decodes 64 packets on one host
    thread for the speedup column (the paper's Table 1 compares its GPU with
    sequential C; context only)."""
    import torch
    import oracle
    from paper_1412_6862_gb300 import hd, synth
    t_setup = time.perf_counter()
    stream = torch.cuda.current_stream(dev)
    sh = stream.cuda_stream
    rows = []
    grid = SHORT_GRID
    if args.short_grid:
        grid = [tuple(int(v) for v in item.split(":")) for item in args.short_grid.split(",")]
    for (M, t) in grid:
        n, k, r = hd.hd_segment_params(M, t)
        P = (SHORT_INPUT_BYTES * 8) // (t * n)
        N = P * t
        seed = M * 10 + t
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        data = torch.randint(-2**31, 2**31 - 1, (hd.words_for(N * k) + 4,), dtype=torch.int32, device=dev,
                             generator=gen)
        enc = hd.encode_short(data, n, N)
        del data
        host = enc.cpu().numpy().view(np.uint32).copy()
        synth.apply_errors(host, synth.error_events(seed, n, N, p1=SHORT_P1, p2=SHORT_P2))
        enc.copy_(torch.from_numpy(host.view(np.int32)))
        out = torch.empty(hd.words_for(N * k) + 4, dtype=torch.int32, device=dev)
        syn = torch.empty(N + 16, dtype=torch.int16, device=dev)
        cnt = torch.empty(2, dtype=torch.int64, device=dev)
        variant = -1 if args.short_no_autotune else hd.hd_short_autotune(n, N, 2, stream)  # at full size, > L2

        def go():
            rc = hd.hd_decode_short(enc.data_ptr(), N * n, n, N, out.data_ptr(), syn.data_ptr(), hd.SYN_U16,
                                    cnt.data_ptr(), cnt.data_ptr() + 8, sh)
            if rc != 0:
                raise hd.HDError(rc, "hd_decode_short")

        for _ in range(3):
            go()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        a.record(stream)
        for _ in range(args.short_steps):
            go()
        b.record(stream)
        torch.cuda.synchronize(dev)
        sec = a.elapsed_time(b) / 1e3 / args.short_steps
        nbytes = N * n / 8 + N * k / 8 + 2 * N
        # oracle: 64 packets (64 t segments) on one host thread
        Po = 64
        o0 = time.perf_counter()
        oracle.decode_short(host, n, Po * t, oracle.SYN_U16)
        o_sec = time.perf_counter() - o0
        counts = cnt.cpu().tolist()
        rows.append({"M": M, "t": t, "n": n, "k": k, "r": r, "packets": P, "segments": N,
                     "us_per_launch": sec * 1e6, "gbps": N * k / sec / 1e9, "packets_per_s": P / sec,
                     "hbm_frac": nbytes / sec / 1e9 / peak, "tile_config": variant,
                     "err_count": counts[0], "detected": counts[1],
                     "speedup_vs_oracle_1thread": (o_sec / Po) / (sec / P)})
        del enc, out, syn, host
        torch.cuda.empty_cache()
    fr = [x["hbm_frac"] for x in rows]
    return {"workload": f"paper (M, t) grid: packets of M in {{400..2000}} bytes cut into t in {{2..6}} segments "
                        f"(shortened Hamming codes, n = 544..8013), ~{SHORT_INPUT_BYTES >> 20} MB of segments per "
                        f"configuration, one hd_decode_short launch each, p1={SHORT_P1}, p2={SHORT_P2} per "
                        f"segment, u16 syndromes",
            "hbm_frac_min": min(fr), "hbm_frac_mean": sum(fr) / len(fr), "hbm_frac_max": max(fr),
            "grid": rows, "setup_s": time.perf_counter() - t_setup}


def l2_bytes(dev):
    import torch
    try:
        return int(torch.cuda.get_device_properties(dev).L2_cache_size)
    except Exception:
        return 126 << 20


def rotation_sets(footprint, dev, floor=2, cap=8):
    """Buffer sets whose total is at least three times the L2, so that a launch
    finds none of its inputs or outputs still in L2 from the launch before."""
    need = (3 * l2_bytes(dev) + footprint - 1) // max(1, footprint)
    return int(max(floor, min(cap, need)))


def time_graph(dev, calls, rounds, warm=2):
    """Capture `calls` (one launch each) `rounds` times over in one CUDA graph,
    replay it `warm` times untimed and once timed with CUDA events on the
    stream it runs on; returns seconds per call."""
    import torch
    stream = torch.cuda.Stream(dev)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        for c in calls:  # warm-up outside the capture (first-use set-up of the library)
            c(stream.cuda_stream)
        torch.cuda.synchronize(dev)
        with torch.cuda.graph(g, stream=stream):
            for _ in range(rounds):
                for c in calls:
                    c(stream.cuda_stream)
        for _ in range(warm):
            g.replay()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        a.record(stream)
        g.replay()
        b.record(stream)
    torch.cuda.synchronize(dev)
    del g
    return a.elapsed_time(b) / 1e3 / (rounds * len(calls))


# (n, syndrome type) -> the autotuner's choice in this process
TUNED = {}


# Every benchmark configuration of a single code (the codes and error rates the
# workload names): (label, n, codewords, [(p1, p2)], syndrome bytes).
PER_CODE = (
    ("Hamming(7,4), 2^20 codewords, p1=0.1, u8 syndromes", 7, 1 << 20, ((0.1, 0.0),), 1),
    ("Hamming(15,11), 2^24 codewords, u8 syndromes", 15, 1 << 24, ((0.01, 0.01), (0.1, 0.01), (0.5, 0.01)), 1),
    ("Hamming(31,26), 2^24 codewords, u8 syndromes", 31, 1 << 24, ((0.01, 0.01), (0.1, 0.01), (0.5, 0.01)), 1),
    ("Hamming(63,57), 2^24 codewords, u8 syndromes", 63, 1 << 24, ((0.01, 0.01), (0.1, 0.01), (0.5, 0.01)), 1),
    ("Hamming(127,120), 2^22 codewords, p1=0.05, p2=0.005, u16 syndromes", 127, 1 << 22, ((0.05, 0.005),), 2),
    ("Hamming(255,247), 2^22 codewords, p1=0.05, p2=0.005, u16 syndromes", 255, 1 << 22, ((0.05, 0.005),), 2),
)


def run_per_code(dev, args, peak):
    """Each code of the workload alone, at every error rate it names: hd_decode
    launches replayed from a CUDA graph over rotating buffer sets (three times
    the L2 in total, so every launch streams from HBM), except (7,4) at 2^20
    codewords, whose 2.5 MB stay in L2 by design and which is reported per
    launch.  The error count is checked against the injected events (every
    event of weight 1 or 2 gives a nonzero syndrome)."""
    import torch
    from paper_1412_6862_gb300 import hd, synth
    res = []
    codes = {int(c) for c in args.per_code_codes.split(",")} if args.per_code_codes else None
    stream = torch.cuda.current_stream(dev)
    for label, n, N, rates, sb in PER_CODE:
        if codes is not None and n not in codes:
            continue
        m, k = code_params(n)
        syn_t = hd.SYN_U8 if sb == 1 else hd.SYN_U16
        # hd_autotune on this code, size and syndrome type (kept from the sweep when already tuned)
        if not args.no_autotune and (n, syn_t) not in TUNED:
            TUNED[(n, syn_t)] = hd.hd_autotune(n, syn_t, N, 5, stream)
        cfg = hd.hd_variant_current(n, syn_t)
        gen = torch.Generator(device=dev)
        gen.manual_seed(2000 + n)
        data = torch.randint(-2**31, 2**31 - 1, (hd.words_for(N * k) + 4,), dtype=torch.int32, device=dev,
                             generator=gen)
        clean = hd.encode(data, n, N).cpu().numpy().view(np.uint32).copy()
        del data
        nbytes = algorithmic_bytes(n, N, sb)
        l2_resident = N * n // 8 < l2_bytes(dev) // 16
        for p1, p2 in rates:
            host = clean.copy()
            ev = synth.error_events(3000 + n, n, N, p1=p1, p2=p2)
            synth.apply_errors(host, ev)
            d0 = torch.from_numpy(host.view(np.int32)).to(dev)
            nsets = 1 if l2_resident else rotation_sets(nbytes, dev)
            sets = []
            for i in range(nsets):
                d_in = d0 if i == 0 else d0.clone()
                out = torch.empty(hd.words_for(N * k) + 4, dtype=torch.int32, device=dev)
                syn = torch.empty(N * sb + 16, dtype=torch.uint8, device=dev)
                err = torch.empty(1, dtype=torch.int64, device=dev)
                sets.append((d_in, out, syn, err))

            def call(bset):
                d_in, out, syn, err = bset
                return lambda sh: hd.check(hd.hd_decode(d_in.data_ptr(), N * n, n, N, out.data_ptr(),
                                                        syn.data_ptr(), syn_t, err.data_ptr(), sh), "hd_decode")

            rounds = 100 if l2_resident else max(2, 12 // nsets)
            t = time_graph(dev, [call(b) for b in sets], rounds)
            errs = [int(b[3].item()) for b in sets]
            res.append({"config": label, "n": n, "codewords": N, "p1": p1, "p2": p2,
                        "kernel": {key: cfg[key] for key in ("threads", "stages", "codewords_per_thread", "inplace",
                                                             "table_lookup")},
                        "us_per_launch": t * 1e6, "gbps": N * k / t / 1e9, "hbm_frac": nbytes / t / 1e9 / peak,
                        "algorithmic_bytes": nbytes, "buffer_sets": nsets, "l2_resident": bool(l2_resident),
                        "err_count": errs[0], "injected_events": int(ev.num_events),
                        "err_count_matches_events": all(e == ev.num_events for e in errs)})
            del sets, d0, host
            torch.cuda.empty_cache()
    return {"workload": "each code alone at every error rate the configurations name; hd_decode replayed from a "
                        "CUDA graph over rotating buffer sets (>= 3x L2 in total) except the L2-resident (7,4) "
                        "stream, whose per-launch time is reported as such", "rows": res}


SECDED_P1, SECDED_P2 = 0.05, 0.005


def run_secded(dev, args, peak):
    """SECDED (extended Hamming, not in the paper) against the plain decoder on
    the same code lengths: 2^24 codewords (n <= 63) or 2^22 (n >= 127), GPU
    encoder, p1/p2 channel errors over the n + 1 bits, u16 syndromes; each
    decoder's launches replayed from a CUDA graph over rotating buffer sets of
    at least three times the L2.  Algorithmic bytes per codeword:
    (n+1)/8 + k/8 + 2 (SECDED), n/8 + k/8 + 2 (plain)."""
    import torch
    from paper_1412_6862_gb300 import hd, synth
    res = {}
    for n in (int(c) for c in args.secded_codes.split(",")):
        m, k = hd.code_params(n)
        N = (1 << 24) if n <= 63 else (1 << 22)
        gen = torch.Generator(device=dev)
        gen.manual_seed(1000 + n)
        data = torch.randint(-2**31, 2**31 - 1, (hd.words_for(N * k) + 4,), dtype=torch.int32, device=dev,
                             generator=gen)
        enc = hd.encode_secded(data, n, N)
        host = enc.cpu().numpy().view(np.uint32).copy()
        synth.apply_errors(host, synth.error_events(1000 + n, n + 1, N, p1=SECDED_P1, p2=SECDED_P2))
        enc.copy_(torch.from_numpy(host.view(np.int32)))
        plain = hd.encode(data, n, N)
        del data, host
        bx = N * (n + 1) / 8 + N * k / 8 + 2 * N
        bp = N * n / 8 + N * k / 8 + 2 * N
        nsets = rotation_sets(int(bx), dev)
        sets = []
        for i in range(nsets):
            sets.append((enc if i == 0 else enc.clone(), plain if i == 0 else plain.clone(),
                         torch.empty(hd.words_for(N * k) + 4, dtype=torch.int32, device=dev),
                         torch.empty(N + 16, dtype=torch.int16, device=dev),
                         torch.empty(2, dtype=torch.int64, device=dev)))

        def go_x(b):
            return lambda sh: hd.check(hd.hd_decode_secded(b[0].data_ptr(), N * (n + 1), n, N, b[2].data_ptr(),
                                                           b[3].data_ptr(), hd.SYN_U16, b[4].data_ptr(),
                                                           b[4].data_ptr() + 8, sh), "hd_decode_secded")

        def go_p(b):
            return lambda sh: hd.check(hd.hd_decode(b[1].data_ptr(), N * n, n, N, b[2].data_ptr(), b[3].data_ptr(),
                                                    hd.SYN_U16, b[4].data_ptr(), sh), "hd_decode")

        rounds = max(2, 12 // nsets)
        tx = time_graph(dev, [go_x(b) for b in sets], rounds)
        counts = sets[0][4].cpu().tolist()
        tp = time_graph(dev, [go_p(b) for b in sets], rounds)
        res[str(n)] = {"codewords": N, "secded_us": tx * 1e6, "secded_gbps": N * k / tx / 1e9,
                       "secded_hbm_frac": bx / tx / 1e9 / peak, "plain_us": tp * 1e6,
                       "plain_gbps": N * k / tp / 1e9, "plain_hbm_frac": bp / tp / 1e9 / peak,
                       "err_count": counts[0], "detected": counts[1], "buffer_sets": nsets}
        del enc, plain, sets
        torch.cuda.empty_cache()
    return {"workload": f"SECDED (extended Hamming, overall parity at position 0) vs plain Hamming, 2^24 "
                        f"codewords (n <= 63) or 2^22 (n >= 127), p1={SECDED_P1}, p2={SECDED_P2} per codeword, "
                        f"u16 syndromes; hd_decode_secded / hd_decode replayed from a CUDA graph over rotating "
                        f"buffer sets (>= 3x L2)", "codes": res}


def serve_rates(args):
    """The named rates, then doubling rates until the server saturates."""
    base = [float(r) for r in args.serve_rates.split(",")]
    extra = [float(r) for r in args.serve_saturation_rates.split(",")] if args.serve_saturation_rates else []
    return base, extra


def run_serving(dev, args, pool=None, host=False):
    """Open-loop Poisson arrivals of packets from the batched distribution,
    served with continuous batching under a 4 GB admission budget: p50/p99
    latency and sustained Gbit/s per arrival rate, then higher rates until the
    sustained rate falls below 90 % of the offered one or arrivals have to
    wait for queue room (saturation).  host=False: payloads pre-staged in
    device memory, arrival = descriptor enqueue.  host=True: payloads and
    results in pinned host memory (hd_serve_trace_host), so the latency
    includes the gather and scatter copies; per-wave stage times (T_PS, T_DKE,
    T_PR) are reported beside Eq. 1 and its slowest-stage form."""
    import torch
    from paper_1412_6862_gb300 import hd, synth
    t_setup = time.perf_counter()
    layout, d_in, d_out, d_syn = pool if pool is not None else build_batched(dev, args.batched_packets)
    P = len(layout)
    if host:
        h_in = d_in.cpu().pin_memory()
        h_out = torch.empty(d_out.numel(), dtype=torch.int32).pin_memory()
        h_syn = torch.empty(d_syn.numel(), dtype=torch.uint8).pin_memory()
        bi, bo, bs = h_in.data_ptr(), h_out.data_ptr(), h_syn.data_ptr()
    else:
        bi, bo, bs = d_in.data_ptr(), d_out.data_ptr(), d_syn.data_ptr()
    rows = [(bi + 4 * oi, bo + 4 * oo, bs + osy, N, n, hd.SYN_U8) for (n, N, oi, oo, osy, od, iw, ow, dw) in layout]
    bits = [N * code_params(n)[1] for (n, N, *_r) in layout]
    num = args.serve_packets
    table = hd.packet_table([rows[j % P] for j in range(num)])
    # host waves also copy their packets in and out: fewer packets per wave
    # keep one wave's copies short (a wave takes whatever is waiting)
    staging = (64 << 20) if host else 0
    wave_packets = 512 if host else 4096
    cfg = hd.server_config(max_waves=4, max_wave_packets=wave_packets, max_wave_tiles=1 << 16,
                           queue_capacity=max(1 << 16, num), mem_cap_bytes=4 << 30, host_staging_bytes=staging)
    setup_s = time.perf_counter() - t_setup
    src = "pinned host memory (gather, decode and scatter per wave on the slot's stream)" if host else \
        "a device pool (arrival = descriptor enqueue)"
    out = {"workload": f"open-loop Poisson arrivals of packets from the batched distribution ({P}-packet pool in "
                       f"{src}, cycled), {num} packets per rate; continuous batching with 4 wave slots, <= "
                       f"{wave_packets} packets per wave{', 64 MB of staging per slot' if host else ''}, 4 GB "
                       f"admission budget; latency = scheduled arrival -> completion seen by the host",
           "setup_s": setup_s, "rates": {}}
    base, extra = serve_rates(args)
    best, saturated_at = 0.0, None
    for i, rate in enumerate(base + extra):
        if i >= len(base) and saturated_at is not None:
            break
        arr = synth.poisson_arrivals(int(rate) % 1000003, num, rate)
        comps, st = hd.hd_serve_trace(cfg, table, arr, num, host=host)
        bad = sum(1 for j in range(num) if comps[j].status != hd.HD_OK)
        decoded = sum(bits[j % P] for j in range(num))
        sustained = decoded / st["duration_s"] / 1e9 if st["duration_s"] > 0 else None
        offered = decoded / float(arr[-1]) / 1e9
        row = {"p50_latency_us": st["p50_latency_us"], "p99_latency_us": st["p99_latency_us"],
               "p999_latency_us": st["p999_latency_us"], "max_latency_us": st["max_latency_us"],
               "max_submit_lag_us": st["max_submit_lag_us"], "sustained_gbps": sustained, "offered_gbps": offered,
               "duration_s": st["duration_s"], "waves": st["waves"], "mean_wave_packets": st["mean_wave_packets"],
               "max_resident_gb": st["max_resident_bytes"] / 1e9, "backpressure_waits": st["backpressure_waits"],
               "failed_packets": bad}
        if host and st["host_waves"]:
            tp, tk, tr = st["mean_t_in_us"] * 1e-6, st["mean_t_decode_us"] * 1e-6, st["mean_t_out_us"] * 1e-6
            w = st["host_waves"]
            row.update({"t_ps_us": tp * 1e6, "t_dke_us": tk * 1e6, "t_pr_us": tr * 1e6,
                        "eq1_prediction": eq1_speedup(w, tp, tk, tr),
                        "slowest_stage_prediction": pipeline_speedup(w, tp, tk, tr),
                        "overlap": w * (tp + tk + tr) / st["duration_s"] if st["duration_s"] > 0 else None})
        out["rates"][f"{rate:g}"] = row
        if sustained:
            best = max(best, sustained)
        if saturated_at is None and (st["backpressure_waits"] > 0 or (sustained or 0) < 0.9 * offered):
            saturated_at = rate
    out["saturation"] = {"max_sustained_gbps": best, "saturated_at_rate": saturated_at,
                         "rule": "the first rate whose sustained Gbit/s fell below 90 % of the offered load or "
                                 "whose arrivals waited for queue room"}
    if host and "rates" in out:
        out["note"] = ("overlap = waves x (T_PS + T_DKE + T_PR) / duration: the mean number of wave stages in "
                       "flight at once, the achieved counterpart of the two predictions")
    return out


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------
ADT_CHUNK = 1 << 21  # codewords per packet of the transfer model (the host pipeline's chunk)


def eq1_speedup(npk, t_ps, t_dke, t_pr):
    """Eq. 1: speedup of ADT over SDT for npk packets, N(T_PS+T_DKE+T_PR) /
    (T_PS + N T_DKE + T_PR): the pipeline hides every packet's transfers behind
    the kernels of the others, i.e. assumes the kernel is the slowest stage."""
    return npk * (t_ps + t_dke + t_pr) / (t_ps + npk * t_dke + t_pr)


def pipeline_speedup(npk, t_ps, t_dke, t_pr):
    """The same three-stage pipeline with the slowest stage S = max(T_PS, T_DKE,
    T_PR) setting the pace: N(T_PS+T_DKE+T_PR) / (T_PS+T_DKE+T_PR + (N-1) S).
    Equals Eq. 1 when the kernel is the slowest stage."""
    s = max(t_ps, t_dke, t_pr)
    return npk * (t_ps + t_dke + t_pr) / (t_ps + t_dke + t_pr + (npk - 1) * s)


def run_adt(bufs, codes, reps=5):
    """The paper's synchronous vs asynchronous data transfer (Sec. III-B, Eq. 1) on
    each sweep stream: the stream is cut into N packets of ADT_CHUNK codewords.
    SDT = every packet's host-to-device copy, decode and device-to-host copy back
    to back on one stream (CUDA events between the stages give the per-packet
    T_PS, T_DKE and T_PR); ADT = hd_decode_host, the library's overlapped
    pipeline, on the whole stream.  Eq. 1 predicts N(T_PS+T_DKE+T_PR) /
    (T_PS + N T_DKE + T_PR), which assumes the kernel is the slowest stage; the
    same pipeline with the slowest stage S = max(T_PS, T_DKE, T_PR) in that place
    gives N(T_PS+T_DKE+T_PR) / (T_PS + T_DKE + T_PR + (N-1) S)."""
    import torch
    from paper_1412_6862_gb300 import hd
    st = torch.cuda.Stream()
    res = {}
    for n in codes:
        b = bufs[n]
        N, k = b["N"], b["k"]
        npk = N // ADT_CHUNK
        iw, ow = ADT_CHUNK * n // 32, ADT_CHUNK * k // 32
        d_in, out, syn, err = b["d_in"], b["out"], b["syn"], b["err"]
        pinned, out_h, syn_h = b["pinned"], b["out_h"], b["syn_h"]
        stage = {"ps": [], "dke": [], "pr": []}
        sdt = []
        for r in range(reps + 1):  # the first round warms up
            evs = []
            with torch.cuda.stream(st):
                for c in range(npk):
                    e = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
                    e[0].record(st)
                    d_in[c * iw:(c + 1) * iw].copy_(pinned[c * iw:(c + 1) * iw], non_blocking=True)
                    e[1].record(st)
                    rc = hd.hd_decode(d_in.data_ptr() + 4 * c * iw, ADT_CHUNK * n, n, ADT_CHUNK,
                                      out.data_ptr() + 4 * c * ow, syn.data_ptr() + c * ADT_CHUNK, hd.SYN_U8,
                                      err.data_ptr(), st.cuda_stream)
                    if rc != 0:
                        raise hd.HDError(rc, "hd_decode")
                    e[2].record(st)
                    out_h[c * ow:(c + 1) * ow].copy_(out[c * ow:(c + 1) * ow], non_blocking=True)
                    syn_h[c * ADT_CHUNK:(c + 1) * ADT_CHUNK].copy_(syn[c * ADT_CHUNK:(c + 1) * ADT_CHUNK],
                                                                   non_blocking=True)
                    e[3].record(st)
                    evs.append(e)
            st.synchronize()
            if r == 0:
                continue
            sdt.append(evs[0][0].elapsed_time(evs[-1][3]) / 1e3)
            for e in evs:
                stage["ps"].append(e[0].elapsed_time(e[1]) / 1e3)
                stage["dke"].append(e[1].elapsed_time(e[2]) / 1e3)
                stage["pr"].append(e[2].elapsed_time(e[3]) / 1e3)
        adt = []
        for r in range(reps + 1):
            t0 = time.perf_counter()
            rc, _ = hd.hd_decode_host(b["pinned"].data_ptr(), N * n, n, N, out_h.data_ptr(), syn_h.data_ptr(),
                                      hd.SYN_U8, ADT_CHUNK)
            if rc != 0:
                raise hd.HDError(rc, "hd_decode_host")
            if r > 0:
                adt.append(time.perf_counter() - t0)
        t_ps, t_dke, t_pr = (float(np.median(stage[x])) for x in ("ps", "dke", "pr"))
        t_sdt, t_adt = float(np.median(sdt)), float(np.median(adt))
        res[str(n)] = {
            "packets": npk, "codewords_per_packet": ADT_CHUNK,
            "t_ps_us": t_ps * 1e6, "t_dke_us": t_dke * 1e6, "t_pr_us": t_pr * 1e6,
            "sdt_ms": t_sdt * 1e3, "adt_ms": t_adt * 1e3, "speedup": t_sdt / t_adt,
            "eq1_prediction": eq1_speedup(npk, t_ps, t_dke, t_pr),
            "slowest_stage_prediction": pipeline_speedup(npk, t_ps, t_dke, t_pr),
        }
    return {"workload": "each sweep stream as N packets of 2^21 codewords: SDT (copy in, decode, copy out, "
                        "per packet, one stream) vs ADT (hd_decode_host, overlapped pipeline); medians of "
                        f"{reps} runs; host buffers pinned", "codes": res}


def section_summary(sections):
    """One figure or two of every section that ran, four digits each."""
    def short(x):
        return float(f"{x:.4g}") if isinstance(x, float) else x

    res = {}
    for name, sec in sections.items():
        if not sec:
            continue
        if name == "batched":
            res[name] = {key: short(sec["persistent_graph"][key]) for key in ("gbps", "hbm_frac", "variant")}
        elif name in ("serving", "serving_host"):
            res[name] = {key: short(v) for key, v in sec.get("saturation", {}).items()
                         if key in ("max_sustained_gbps", "saturated_at_rate")}
        elif name == "shortened":
            res[name] = {key: short(sec[key]) for key in ("hbm_frac_min", "hbm_frac_mean", "hbm_frac_max")}
        elif name == "secded":
            res[name] = {n: short(row["secded_hbm_frac"]) for n, row in sec["codes"].items()}
        elif name == "per_code":
            fr = [row["hbm_frac"] for row in sec["rows"] if not row["l2_resident"]]
            res[name] = {"hbm_frac_min": short(min(fr)), "hbm_frac_max": short(max(fr))} if fr else {}
        elif name == "adt":
            res[name] = {n: short(row["speedup"]) for n, row in sec["codes"].items()}
    return res


def run_ours(args):
    import torch
    rank, world, local = dist_setup(args.gpus)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    from paper_1412_6862_gb300 import build as hd_build
    hd_build.build()
    from paper_1412_6862_gb300 import hd, synth

    if args.batched_only:
        res = run_batched(dev, args, peaks()[0])
        if rank == 0:
            print(json.dumps({"batched": res}), flush=True)
        return
    if args.serve_only:
        res = run_serving(dev, args)
        res_h = None if args.no_serve_host else run_serving(dev, args, host=True)
        if rank == 0:
            print(json.dumps({"serving": res, "serving_host": res_h}), flush=True)
        return
    if args.secded_only:
        res = run_secded(dev, args, peaks()[0])
        if rank == 0:
            print(json.dumps({"secded": res}), flush=True)
        return
    if args.shortened_only:
        res = run_shortened(dev, args, peaks()[0])
        if rank == 0:
            print(json.dumps({"shortened": res}), flush=True)
        return
    if args.per_code_only:
        res = run_per_code(dev, args, peaks()[0])
        if rank == 0:
            print(json.dumps({"per_code": res}), flush=True)
        return

    codes = tuple(int(c) for c in args.codes.split(","))
    assert all(c in SWEEP_CODES for c in codes), codes
    roof_n = ROOFLINE_N if ROOFLINE_N in codes else max(codes)
    stream_h = torch.cuda.current_stream(dev)
    sh = int(stream_h.cuda_stream)
    bufs = {}
    for n in codes:
        m, k = code_params(n)
        N = SWEEP_N
        seed = shard_seed(n, rank)
        data = synth.random_words(seed, N * k)
        d_data = torch.from_numpy(data.view(np.int32)).to(dev)
        d_in = hd.encode(d_data, n, N)                      # GPU encoder builds the codewords
        host = d_in.cpu().numpy().view(np.uint32).copy()
        synth.apply_errors(host, synth.error_events(seed, n, N, p1=SWEEP_P1, p2=SWEEP_P2))
        pinned = torch.from_numpy(host.view(np.int32)).pin_memory()
        d_in.copy_(pinned)
        del d_data
        out = torch.empty(hd.words_for(N * k), dtype=torch.int32, device=dev)
        syn = torch.empty(N, dtype=torch.uint8, device=dev)
        err = torch.empty(1, dtype=torch.int64, device=dev)
        out_h = torch.empty_like(out, device="cpu").pin_memory()
        syn_h = torch.empty_like(syn, device="cpu").pin_memory()
        err_h = torch.empty_like(err, device="cpu").pin_memory()
        bufs[n] = dict(N=N, k=k, d_in=d_in, pinned=pinned, out=out, syn=syn, err=err,
                       out_h=out_h, syn_h=syn_h, err_h=err_h)
    torch.cuda.synchronize()

    # hd_autotune times every compiled configuration of each code at the
    # sweep's size on random data streamed from HBM (outside the timed region)
    # and keeps the fastest, unless the built-in one is within its noise margin
    tuned = {}
    pins = dict(tuple(int(v) for v in item.split(":")) for item in args.pin.split(",")) if args.pin else {}
    for n in codes:
        if n in pins:
            hd.hd_variant_select(n, hd.SYN_U8, pins[n])
            info = hd.hd_variant_current(n, hd.SYN_U8)
        elif not args.no_autotune:
            info = hd.hd_autotune(n, hd.SYN_U8, SWEEP_N, 5, stream_h)
            TUNED[(n, hd.SYN_U8)] = info
        else:
            continue
        tuned[str(n)] = {key: info[key] for key in ("threads", "stages", "codewords_per_thread", "inplace",
                                                    "table_lookup")}
    torch.cuda.synchronize()

    def decode_call(n, cuda_stream):
        b = bufs[n]
        rc = hd.hd_decode(b["d_in"].data_ptr(), n * b["N"], n, b["N"], b["out"].data_ptr(), b["syn"].data_ptr(),
                          hd.SYN_U8, b["err"].data_ptr(), cuda_stream)
        if rc != 0:
            raise hd.HDError(rc, "hd_decode")

    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    for _ in range(args.warmup):
        for n in codes:
            decode_call(n, sh)
    barrier()

    # One step = one hd_decode_streams call captured in a CUDA graph: the
    # counters are cleared by one kernel, then the codes' decodes run as
    # concurrent branches (the streams are independent, so one decode's fill
    # and drain overlap another's streaming instead of idling SMs)
    jobs = hd.stream_jobs([(bufs[n]["d_in"].data_ptr(), n, bufs[n]["N"], bufs[n]["out"].data_ptr(),
                            bufs[n]["syn"].data_ptr(), hd.SYN_U8, bufs[n]["err"].data_ptr()) for n in codes])

    def step_call(cuda_stream):
        rc = hd.hd_decode_streams(jobs, len(codes), cuda_stream)
        if rc != 0:
            raise hd.HDError(rc, "hd_decode_streams")

    step_call(sh)  # the first call creates the library's branch streams, outside any capture
    torch.cuda.synchronize()
    step_graph = torch.cuda.CUDAGraph()
    cap = torch.cuda.Stream(dev)
    l0 = hd.hd_launch_count()
    with torch.cuda.graph(step_graph, stream=cap):
        step_call(cap.cuda_stream)
    launches_per_step = hd.hd_launch_count() - l0
    for _ in range(3):
        step_graph.replay()
    barrier()

    uuid = None
    try:
        uuid = str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    with ClockSampler(uuid) as clk:
        barrier()
        t_start.record(stream_h)
        for i in range(args.steps):
            step_graph.replay()
        t_end.record(stream_h)
        barrier()
    launches = launches_per_step * args.steps
    ms = reduce_max(t_start.elapsed_time(t_end), dev)
    bits_per_step = sum(bufs[n]["N"] * bufs[n]["k"] for n in codes)
    value = weak_scaling_value(bits_per_step * args.steps, world, ms / 1e3) / 1e9
    roof_bytes = algorithmic_bytes(roof_n, SWEEP_N)
    peak, peak_kind = peaks()
    vinfo = hd.hd_variant_current(roof_n, hd.SYN_U8)
    kernel_desc = (f"k_decode_stream<{roof_n}, 1, {vinfo['threads']}, {vinfo['stages']}, "
                   f"{vinfo['codewords_per_thread']}, {vinfo['inplace']}>")
    traffic = recorded_traffic(kernel_desc) if roof_n == ROOFLINE_N else None
    clocks = clk.summary()
    # the whole step against the same peak: every byte the step's launches
    # move over the step's time
    step_bytes = sum(algorithmic_bytes(n, SWEEP_N) for n in codes)
    step_frac = step_bytes / (ms / args.steps / 1e3) / 1e9 / peak
    # the dominant kernel alone, back to back: ten launches in one graph over
    # two buffer sets (536 MB, more than three times the L2), timed with CUDA
    # events on the stream the graph runs on; each launch also pays for its
    # predecessor's write-back, so nothing leaves the measurement in L2
    b = bufs[roof_n]
    spare = dict(d_in=b["d_in"].clone(), out=torch.empty_like(b["out"]), syn=torch.empty_like(b["syn"]),
                 err=torch.empty_like(b["err"]))

    def roof_call(bs):
        return lambda sh_: hd.check(hd.hd_decode(bs["d_in"].data_ptr(), roof_n * SWEEP_N, roof_n, SWEEP_N,
                                                 bs["out"].data_ptr(), bs["syn"].data_ptr(), hd.SYN_U8,
                                                 bs["err"].data_ptr(), sh_), "hd_decode")

    t_b2b = time_graph(dev, [roof_call(b), roof_call(spare)], 5)
    del spare
    torch.cuda.empty_cache()
    kern_ms = t_b2b * 1e3
    achieved = roof_bytes / t_b2b / 1e9

    # end to end through the C ABI with HOST buffers: hd_decode_host copies each
    # stream from pinned host memory, decodes it and copies data bits,
    # syndromes and err_count back, overlapping the copies with the decode
    h2d = sum(bufs[n]["pinned"].numel() * 4 for n in codes)
    d2h = sum(bufs[n]["out"].numel() * 4 + bufs[n]["syn"].numel() + 8 for n in codes)

    e2e_jobs = [(bufs[n]["pinned"].data_ptr(), n, bufs[n]["N"], bufs[n]["out_h"].data_ptr(),
                 bufs[n]["syn_h"].data_ptr(), hd.SYN_U8) for n in codes]

    def e2e_step():
        # the three streams in one pipeline of host-to-device copies, decodes and
        # device-to-host copies (one fill and one drain per step)
        rc, _ = hd.hd_decode_host_batch(e2e_jobs)
        if rc != 0:
            raise hd.HDError(rc, "hd_decode_host_batch")

    e2e_steps = 0 if args.no_e2e else args.e2e_steps
    for _ in range(3 if e2e_steps else 0):
        e2e_step()
    barrier()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        e2e_step()
    barrier()
    e2e_s = reduce_max(max(time.perf_counter() - t0, 1e-9), dev)
    e2e_value = weak_scaling_value(bits_per_step * e2e_steps, world, e2e_s) / 1e9 if e2e_steps else None
    adt = None if (args.no_adt or args.no_e2e) else run_adt(bufs, codes)

    batched = serving = None
    if not (args.no_batched and args.no_serve):
        for b in bufs.values():  # free the sweep's buffers first
            b.clear()
        bufs.clear()
        torch.cuda.empty_cache()
    pool = None
    if not args.no_batched:
        batched, pool = run_batched(dev, args, peak, keep_pool=True)
    serving_host = None
    if not args.no_serve:
        serving = run_serving(dev, args, pool)
        if not args.no_serve_host:
            serving_host = run_serving(dev, args, pool, host=True)
    pool = None
    shortened = None
    if not args.no_shortened:
        torch.cuda.empty_cache()
        shortened = run_shortened(dev, args, peak)
    secded = None
    if not args.no_secded:
        torch.cuda.empty_cache()
        secded = run_secded(dev, args, peak)
    per_code = None
    if not args.no_per_code:
        torch.cuda.empty_cache()
        per_code = run_per_code(dev, args, peak)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(args.cpu_seconds)

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "Gbit/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {"workload": WORKLOAD if codes == SWEEP_CODES else f"subset {codes} of: {WORKLOAD}",
                       "num_codewords": SWEEP_N, "codes": list(codes),
                       "parallelism": f"replicas{world}" if world > 1 else "single-gpu",
                       "l2": "inputs larger than L2 (475 MB of streams and outputs, each touched once per step)",
                       "step": "one hd_decode_streams call (the three decodes as concurrent branches) in a CUDA graph",
                       "kernel_configs": tuned or "built-in"},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": traffic,
                         "kernel": f"hd_decode n={roof_n}, N=2^24 ({roof_bytes} algorithmic bytes/launch, "
                                   f"{kern_ms * 1e3:.2f} us avg over 10 back-to-back launches; {kernel_desc})",
                         "peak_kind": peak_kind, "step_frac": step_frac, "step_bytes": step_bytes,
                         "note": "achieved: the dominant kernel alone over two buffer sets; step_frac: the whole "
                                 "step's algorithmic bytes over the timed step"},
            "e2e": {"value": e2e_value, "unit": "Gbit/s", "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
            "gpu_launches": int(launches),
            "clocks": clocks,
            "cpu_baseline": cpu,
        }
        sections = {"batched": batched, "serving": serving, "serving_host": serving_host, "shortened": shortened,
                    "secded": secded, "per_code": per_code, "adt": adt}
        print(json.dumps({"sections": sections}), file=sys.stderr, flush=True)
        line["sections"] = section_summary(sections)
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


def main():
    args = parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
