#!/usr/bin/env python
"""Block-tree build throughput on GB300.

One step = one complete bt_build of the workload text (prefix fingerprints,
every level's fingerprint / window-scan / verify / mark / pointer / split pass,
pruning, rank-select counters, leaf text), i.e. the whole hot path, followed by
bt_free.  Default workload: the 256 MiB versioned text (4 MiB Zipf(1.1) base
over 96 symbols, 64 versions with 0.05 % edit runs), tau = 4, leaf_len = 32.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload NAME]
    python bench.py --impl reference ...   # the CPU oracle, as it stands

Prints one JSON line.  `value` is throughput with the text already resident in
HBM; `e2e` is the same metric through the public C ABI with a host buffer (the
host->device copy of the text and the device->host read of the serialized tree
inside the timed region).  With N > 1 (torchrun) every rank builds its own
replica of the workload: the method has no cross-GPU exchange for a single
text, so there is no data-path collective.
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

from paper_2512_23314_gb300 import workloads  # noqa: E402

METRIC = "block tree build MB/s"
UNIT = "MB/s"

WORKLOADS = {
    "text_versions_256MiB": dict(
        gen=lambda: workloads.text_versions(), sigma=96, tau=4, leaf=32,
        desc="256 MiB versioned text: 4 MiB Zipf(1.1) base over 96 symbols, 64 versions "
             "with 0.05% substitute/insert/delete runs of 1-32 bytes"),
    "text_versions_160MiB": dict(
        gen=lambda: workloads.text_versions(n=160 << 20), sigma=96, tau=4, leaf=32,
        desc="160 MiB prefix of the versioned-text workload (profiling captures)"),
    "dna_copies_1MiB": dict(
        gen=lambda: workloads.dna_copies(), sigma=4, tau=2, leaf=16,
        desc="1 MiB DNA: 64 KiB uniform ACGT seed copied 16 times with 0.1% substitutions"),
    "dna_genome_2GiB": dict(
        gen=lambda: workloads.dna_genome(), sigma=5, tau=4, leaf=64,
        desc="2 GiB DNA: 32 MiB uniform ACGT genome, 64 copies with 0.1% SNPs, "
             "0.01% indels of 1-50 bases, N runs",
        opts={"two_phase": True}),
}
DEFAULT_WORKLOAD = "text_versions_256MiB"
HBM_SPEC_GBS = 8000.0  # nominal HBM3e bandwidth of a GB300
SCAN_SOURCE = os.path.join(ROOT, "paper_2512_23314_gb300", "csrc", "bt_level.cu")


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default=DEFAULT_WORKLOAD)
    ap.add_argument("--cpu-sample-mib", type=int, default=8,
                    help="prefix of the workload the CPU oracle builds per step")
    ap.add_argument("--cpu-mt-sample-mib", type=int, default=1 << 20,
                    help="prefix of the workload the multithreaded CPU builder builds (default: all)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the batched-build and serving measurements")
    ap.add_argument("--batch-docs", type=int, default=8192,
                    help="documents of the batched-build measurement (default: the full batched workload)")
    ap.add_argument("--batch-max-mib", type=int, default=16,
                    help="largest document of the batched-build measurement in MiB")
    ap.add_argument("--batch-only", action="store_true",
                    help="run only the batched-build measurement and print its JSON object")
    ap.add_argument("--summarize-launches", metavar="CSV",
                    help="summarize an ncu launch list (--metrics gpu__time_duration.sum --csv) and exit")
    ap.add_argument("--builds", type=int, default=1,
                    help="builds the launch list covers (with --summarize-launches / --summarize-traffic)")
    ap.add_argument("--summarize-traffic", nargs=3, metavar=("CSV", "BENCH_JSON", "OUT_JSON"),
                    help="window-scan DRAM traffic from an ncu capture (--metrics dram__bytes_read.sum,"
                         "dram__bytes_write.sum,gpu__time_duration.sum --csv) of the same build as the "
                         "bench line in BENCH_JSON; writes the traffic record and exits")
    return ap.parse_args()


def summarize_launches(path: str, builds: int) -> None:
    """Per kernel of an ncu launch list: launches, time per build and share of
    the kernel time; then the per-level durations of the window-scan kernels
    of one build (the launch list's second build, after the warm-up)."""
    import collections
    import csv
    rows = [r for r in csv.reader(open(path)) if len(r) > 10]
    hdr, rows = rows[0], rows[1:]
    i_name, i_val = hdr.index("Kernel Name"), hdr.index("Metric Value")
    agg = collections.defaultdict(lambda: [0, 0.0])
    per = collections.defaultdict(list)
    for r in rows:
        name = r[i_name].split("(")[0].replace("void ", "").replace("(anonymous namespace)::", "")
        name = name.replace("unnamed>::", "")
        ms = float(r[i_val].replace(",", "")) / 1e6
        agg[name][0] += 1
        agg[name][1] += ms
        per[name].append(ms)
    tot = sum(v[1] for v in agg.values())
    print(f"launches {sum(v[0] for v in agg.values())}, kernel time {tot / builds:.2f} ms per build")
    print(f"{'kernel':44s} {'launches':>8s} {'ms/build':>9s} {'share':>7s}")
    for k, v in sorted(agg.items(), key=lambda x: -x[1][1])[:40]:
        print(f"{k:44s} {v[0]:8d} {v[1] / builds:9.3f} {100 * v[1] / tot:6.2f}%")
    for k in per:
        if any(s in k for s in ("k_chase_scan", "k_quick_compare", "k_scan_anchor", "k_hits", "k_candidates<")):
            n = len(per[k]) // builds
            lo = n if builds > 1 else 0
            print(k, "per level:", " ".join(f"{x:.3f}" for x in per[k][lo:lo + n]))


SCAN_KERNELS = ("k_scan", "k_hits", "k_candidates<")
TRAFFIC_CMD = ("ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum "
               "--clock-control none -k \"regex:k_scan|k_hits|k_candidates\" --csv --log-file dram.csv "
               "python bench.py --workload text_versions_160MiB --steps 1 --warmup 0 --no-cpu-baseline --no-extras")


def summarize_traffic(csv_path: str, bench_json: str, out_path: str, builds: int) -> None:
    """DRAM bytes of the window-scan kernels per build, from an ncu capture
    of `builds` identical builds, against the algorithmic bytes (the summed
    level coverage) of the bench line of the same workload; written as the
    traffic record that roofline.traffic reads (keyed by the scan source's
    hash).  The prune pass's own candidate kernel (`k_candidates` without a
    template argument) is not part of the window scan."""
    import collections
    import csv
    scale = {"byte": 1, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9, "nsecond": 1e-6, "usecond": 1e-3,
             "msecond": 1.0, "second": 1e3, "ns": 1e-6, "us": 1e-3, "ms": 1.0, "s": 1e3}
    rows = [r for r in csv.reader(open(csv_path)) if len(r) > 10]
    hdr, rows = rows[0], rows[1:]
    i_name, i_metric = hdr.index("Kernel Name"), hdr.index("Metric Name")
    i_unit, i_val = hdr.index("Metric Unit"), hdr.index("Metric Value")
    agg = collections.defaultdict(lambda: {"ids": set(), "dram_read_bytes": 0.0, "dram_write_bytes": 0.0,
                                           "ms": 0.0})
    i_id = hdr.index("ID")
    for r in rows:
        name = r[i_name].split("(")[0].replace("void ", "").replace("(anonymous namespace)::", "")
        name = name.replace("unnamed>::", "").strip()
        if not any(name.startswith(k) for k in SCAN_KERNELS):
            continue
        v = float(r[i_val].replace(",", "")) * scale.get(r[i_unit], 1.0)
        a = agg[name]
        a["ids"].add(r[i_id])
        key = {"dram__bytes_read.sum": "dram_read_bytes", "dram__bytes_write.sum": "dram_write_bytes",
               "gpu__time_duration.sum": "ms"}.get(r[i_metric])
        if key:
            a[key] += v
    line = json.loads(open(bench_json).read().strip().splitlines()[-1])
    alg = line["config"]["sum_cov_bytes"]
    per = {k: {"launches_per_build": len(a["ids"]) // builds,
               "dram_read_bytes": int(a["dram_read_bytes"] / builds),
               "dram_write_bytes": int(a["dram_write_bytes"] / builds),
               "ms": round(a["ms"] / builds, 4)} for k, a in agg.items()}
    dram = sum(p["dram_read_bytes"] + p["dram_write_bytes"] for p in per.values())
    rec = {"kernel": "window_scan", "source": os.path.relpath(SCAN_SOURCE, ROOT),
           "source_sha256_16": source_hash(SCAN_SOURCE),
           "workload": f"{line['config']['workload']} (n = {line['config']['n']}, tau {line['config']['tau']}, "
                       f"leaf {line['config']['leaf_len']}, prune on), {line['config']['levels']} levels",
           "command": TRAFFIC_CMD, "builds_captured": builds, "alg_bytes_per_build": alg, "dram_bytes_per_build": dram,
           "dram_bytes_per_alg_byte": round(dram / alg, 4), "per_kernel": per}
    with open(out_path, "w") as f:
        json.dump(rec, f, indent=1)
    print(json.dumps(rec, indent=1))


def measured_peaks() -> dict:
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except OSError:
        return {}


def source_hash(path: str) -> str:
    with open(path, "rb") as f:
        return hashlib.sha256(f.read()).hexdigest()[:16]


def recorded_traffic(kernel: str) -> float | None:
    """DRAM bytes per algorithmic byte from the committed ncu summary, if it
    was taken on the current kernel source."""
    path = os.path.join(ROOT, "profiles", "window_scan_traffic.json")
    try:
        with open(path) as f:
            rec = json.load(f)
    except OSError:
        return None
    if rec.get("kernel") != kernel or rec.get("source_sha256_16") != source_hash(SCAN_SOURCE):
        return None
    return rec.get("dram_bytes_per_alg_byte")


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.proc = None
        self.file = None

    def start(self):
        try:
            self.file = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=self.file, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self) -> dict | None:
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.file.flush()
        self.file.seek(0)
        rows = [r.split(",") for r in self.file.read().strip().splitlines() if r.strip()]
        os.unlink(self.file.name)
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            r = [x.strip() for x in r]
            if len(r) < 9:
                continue
            try:
                sm.append(float(r[1]))
                mx.append(float(r[2]))
            except ValueError:
                continue
            for nm, v in zip(names, r[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "samples": len(sm),
                "reasons": sorted(reasons)}


def max_over_ranks(x: float, world: int, device: str = "cuda") -> float:
    """Maximum of a per-rank scalar (timings are taken as the slowest rank)."""
    if world <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def throughput_mbs(n_bytes: int, steps: int, world: int, ms: float) -> float:
    """Whole-job MB/s: every rank builds `steps` replicas of an n-byte text."""
    return n_bytes * steps * world / (ms / 1e3) / 1e6


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def cpu_baseline(text: np.ndarray, w: dict, sample_mib: int, steps: int = 1) -> dict:
    """The oracle as it stands, single-threaded, on a prefix of the workload."""
    import oracle
    n = min(len(text), sample_mib << 20)
    sample = np.ascontiguousarray(text[:n])
    times = []
    for _ in range(steps):
        t0 = time.perf_counter()
        oracle.build(sample, w["tau"], w["leaf"], prune=True)
        times.append(time.perf_counter() - t0)
    sec = statistics.median(times)
    return {"value": n / sec / 1e6, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"first {n} bytes ({n >> 20} MiB) of the workload text, prune on, "
                      f"median of {steps} single-threaded builds"}


def measure_queries(bt, torch, stream, h: int, text: np.ndarray, m: int = 4 << 20, reps: int = 3) -> dict:
    """Query throughput of a built tree: m device-resident queries per batch
    (bt_query_batch), each kind timed with CUDA events over `reps` batches
    after one warm-up; the arguments are seeded and uniform (access: i in
    [0, n); rank: a present symbol and i in [0, n]; select: a present symbol
    and j in [1, its count]).  The first 1000 access answers are checked
    against the text."""
    rng = np.random.default_rng(0xB7EE0005)
    n = len(text)
    counts = np.bincount(text, minlength=256)
    syms = np.flatnonzero(counts)
    c = syms[rng.integers(0, len(syms), m)].astype(np.uint64)
    args = {
        bt.BT_Q_ACCESS: rng.integers(0, n, m, dtype=np.uint64),
        bt.BT_Q_RANK: np.stack([c, rng.integers(0, n + 1, m, dtype=np.uint64)], 1).ravel(),
        bt.BT_Q_SELECT: np.stack([c, (rng.random(m) * counts[c.astype(np.int64)]).astype(np.uint64) + 1],
                                 1).ravel(),
    }
    out = torch.empty(m, dtype=torch.int64, device="cuda")
    res = {"queries_per_batch": m, "batches": reps, "args": "seeded uniform, device-resident"}
    for kind, name in ((bt.BT_Q_ACCESS, "access"), (bt.BT_Q_RANK, "rank"), (bt.BT_Q_SELECT, "select")):
        d_args = torch.from_numpy(args[kind].view(np.int64)).cuda()
        bt.bt_query_batch(h, kind, d_args, m, out, stream)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            bt.bt_query_batch(h, kind, d_args, m, out, stream)
        e1.record(stream)
        e1.synchronize()
        res[f"{name}_per_s"] = m * reps / (e0.elapsed_time(e1) / 1e3)
        if kind == bt.BT_Q_ACCESS:
            got = out[:1000].cpu().numpy()
            idx = args[kind][:1000].astype(np.int64)
            res["access_check"] = bool(np.array_equal(got, text[idx].astype(np.int64)))
    return res


def int_roofline(bt, torch, stream, mulmods_per_step: int, step_ms: float, work: str) -> dict:
    """The integer-pipe roofline of the build: the measured rate of the 61-bit
    modular multiply (the library's microbenchmark, 8 CTAs of 256 threads per
    SM, 8 independent chains per thread) against the 61-bit multiplies the
    timed kernels actually issue in a step (`work` says how they are counted)."""
    blocks = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count * 8
    out = torch.empty(blocks * 256, dtype=torch.int64, device="cuda")
    bt.bt_mulmod_bench(blocks, 64, out, stream)  # warm-up
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    n = bt.bt_mulmod_bench(blocks, 4096, out, stream)
    e1.record(stream)
    e1.synchronize()
    rate = n / (e0.elapsed_time(e1) / 1e3)
    t_roof_ms = mulmods_per_step / rate * 1e3
    return {"bound": "alu", "work": work,
            "mulmods_per_step": mulmods_per_step, "peak": rate / 1e12, "unit": "Tmulmod/s",
            "peak_source": f"measured: {n} multiplies in {e0.elapsed_time(e1):.3f} ms",
            "t_roof_ms": t_roof_ms, "frac": t_roof_ms / step_ms if step_ms > 0 else None}


def issued_mulmods(n: int, stats: list[dict]) -> tuple[int, str]:
    """61-bit modular multiplies a build issues: two per text byte for the
    prefix fingerprints (the chunk Horner pass and the expansion to every
    position), one per block for the block fingerprints, one per window the
    anchored scan tests, and one more per window that matches a block (the
    fingerprint of the following block for the pair join; an upper bound,
    since the join is skipped past the slot's last pair start)."""
    blocks = sum(s["nblocks"] for s in stats)
    cands = sum(s["candidates"] for s in stats)
    hits = sum(s["hits"] for s in stats)
    work = ("issued: 2 per text byte (prefix fingerprints) + 1 per block + 1 per tested window "
            "+ 1 per window matching a block (pair join, upper bound)")
    return 2 * n + blocks + cands + hits, work


def cpu_mt_baseline(text: np.ndarray, w: dict, sample_mib: int) -> dict:
    """The straightforward multithreaded CPU builder (OpenMP, every host core)
    on a prefix of the workload: the multicore CPU baseline."""
    import cpu_mt
    n = min(len(text), sample_mib << 20)
    sample = np.ascontiguousarray(text[:n])
    try:
        t0 = time.perf_counter()
        cpu_mt.build_tree(sample, w["tau"], w["leaf"], prune=True)
        sec = time.perf_counter() - t0
    except (OSError, RuntimeError, subprocess.CalledProcessError) as e:
        return {"unavailable": f"multithreaded CPU builder failed: {e}"}
    return {"value": n / sec / 1e6, "unit": UNIT, "cores": cpu_mt.threads(), "kind": "cpu_mt",
            "sample": f"first {n} bytes ({n >> 20} MiB) of the workload text, prune on, "
                      f"one OpenMP build on {cpu_mt.threads()} threads"}


def measure_batch(ndocs: int = 8192, min_len: int = 4 << 10, max_len: int = 16 << 20,
                  nworkers: int = 16) -> dict:
    """The batched workload: `ndocs` versioned-text documents of log-uniform
    length (4 KiB - 16 MiB by default: 8192 documents, ~16.5 GB), sigma
    4-128, tau 2/4/8, leaf 32.  Three arms, the texts in one pinned host
    buffer in each (the copy to the device is inside every timed call):
      plain   -- one bt_build_ex call per document, back to back (one
                 document per launch sequence);
      workers -- bt_build_batch with BT_FLAG_BATCH_WORKERS (bt_build_ex on
                 host threads, one CUDA stream each);
      kernel  -- bt_build_batch: the persistent batched kernel.
    Each arm is timed once after a warm-up batch; the exports of a seeded
    sample of documents are compared between the arms."""
    import torch

    from paper_2512_23314_gb300 import bt
    t_gen = time.perf_counter()
    docs = workloads.doc_mix(ndocs, min_len=min_len, max_len=max_len, seed=0xB7EE0004)
    gen_s = time.perf_counter() - t_gen
    pinned = torch.empty(sum(len(d.text) for d in docs), dtype=torch.uint8, pin_memory=True)
    texts, o = [], 0
    for d in docs:
        v = pinned[o:o + len(d.text)]
        v.copy_(torch.from_numpy(d.text))
        texts.append(v)
        o += len(d.text)
    args = (texts, [len(d.text) for d in docs], [d.sigma for d in docs],
            [d.tau for d in docs], [d.leaf_len for d in docs])
    sample = sorted(np.random.default_rng(7).choice(ndocs, min(64, ndocs), replace=False).tolist())
    o_kernel, _ = bt.BuildOptions().to_c()
    o_workers, _ = bt.BuildOptions(batch_workers=True).to_c()

    def batch_arm(o):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        hs = bt.bt_build_batch(*args, o, nworkers=nworkers)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        blobs = [hashlib.sha256(bt.bt_export(hs[i])).hexdigest() for i in sample]
        rep = bt.bt_batch_report()
        cyc = np.array([bt.bt_batch_cycles(h) for h in hs], dtype=np.float64)
        for h in hs:
            bt.bt_free(h)
        return dt, blobs, rep, cyc

    # Warm-up on the whole batch (the first call maps its memory).
    warm = bt.bt_build_batch(*args, o_kernel, nworkers=nworkers)
    for h in warm:
        bt.bt_free(h)
    kernel_s, kernel_blobs, rep, cyc = batch_arm(o_kernel)
    workers_s, workers_blobs, _, _ = batch_arm(o_workers)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    plain_blobs = {}
    for i, d in enumerate(docs):
        h = bt.bt_build_ex(texts[i], len(d.text), d.sigma, d.tau, d.leaf_len)
        if i in sample:
            plain_blobs[i] = hashlib.sha256(bt.bt_export(h)).hexdigest()
        bt.bt_free(h)
    torch.cuda.synchronize()
    plain_s = time.perf_counter() - t0
    same = kernel_blobs == workers_blobs == [plain_blobs[i] for i in sample]
    total = sum(len(d.text) for d in docs)
    phases = ["setup", "tables", "window_scan", "verify_mark_split", "prune", "output_counters"]
    share = (cyc.sum(0) / cyc.sum()).tolist() if cyc.sum() > 0 else None
    return {"workload": f"{ndocs} versioned-text documents, log-uniform {min_len >> 10} KiB - "
                        f"{max_len >> 20} MiB, sigma 4-128, tau 2/4/8, leaf 32; texts in pinned host memory",
            "generate_s": gen_s, "docs": ndocs, "bytes": total,
            "docs_per_s": ndocs / kernel_s, "mb_per_s": total / kernel_s / 1e6,
            "kernel_device_mb_per_s": total / (rep["kernel_us"] * 1e-6) / 1e6 if rep["kernel_us"] else None,
            "workers_docs_per_s": ndocs / workers_s, "plain_docs_per_s": ndocs / plain_s,
            "speedup_vs_plain": plain_s / kernel_s, "speedup_vs_workers": workers_s / kernel_s,
            "workers_mb_per_s": total / workers_s / 1e6, "plain_mb_per_s": total / plain_s / 1e6,
            "identical_output_sample": {"docs": len(sample), "equal": bool(same)},
            "kernel": rep,
            "kernel_phase_share": dict(zip(phases, share)) if share else None,
            "nworkers": nworkers}


def measure_sort_variant(bt, torch, stream, d_text, n, w, blob) -> dict:
    """The sort-based level pass (section 4.1) on the headline text, as one
    part and in K parts (the domain decomposition of section 4.2), beside the
    default anchored scan: build time and the peak of the device pool during
    the build (the working memory).  One warm-up and one timed build each."""
    out = {"parts": {}}

    def timed(opts):
        o = bt.BuildOptions(prune=True, **opts, **w.get("opts", {})).to_c()[0]
        bt.bt_free(bt.bt_build_ex(d_text, n, w["sigma"], w["tau"], w["leaf"], o, stream))
        torch.cuda.synchronize()
        bt.bt_device_pool_peak(reset=True)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        h = bt.bt_build_ex(d_text, n, w["sigma"], w["tau"], w["leaf"], o, stream)
        e1.record(stream)
        torch.cuda.synchronize()
        peak = bt.bt_device_pool_peak()
        same = bt.bt_export(h) == blob
        bt.bt_free(h)
        ms = e0.elapsed_time(e1)
        return {"ms": ms, "mb_per_s": n / (ms * 1e-3) / 1e6, "peak_pool_bytes": peak,
                "peak_bytes_per_text_byte": peak / n, "same_export": same}

    out["default_anchored"] = timed({})
    for k in (1, 4, 16):
        out["parts"][str(k)] = timed({"sort_scan": True, "partitions": k})
    return out


def measure_serve(rate: float = 2000.0, duration: float = 0.5, min_len: int = 1 << 10,
                  max_len: int = 64 << 20, lanes: int = 8, small_max: int = 1 << 20) -> dict:
    """The serving loop over the serving workload's full length range (1 KiB -
    64 MiB, DNA-like / text-like 50/50, 120 GiB budget, 10^4 queries per
    document), with a 0.5 s window of Poisson arrivals at 2000 documents/s
    (the 10 s stream would offer ~120 GB of text, too much to generate within
    a bench run).  Documents up to 1 MiB are built in micro-batches by the
    batched kernel, larger ones alone.  The texts arrive in pinned host
    memory, as a server's receive buffers would hold them."""
    import torch

    from paper_2512_23314_gb300 import serve
    t0 = time.perf_counter()
    arrivals = workloads.serve_arrivals(rate=rate, duration=duration, min_len=min_len,
                                        max_len=max_len)
    pinned = torch.empty(sum(len(a.doc.text) for a in arrivals), dtype=torch.uint8, pin_memory=True)
    staged, o = [], 0
    for a in arrivals:
        v = pinned[o:o + len(a.doc.text)]
        v.copy_(torch.from_numpy(a.doc.text))
        staged.append(workloads.Arrival(a.t, workloads.Doc(v, a.doc.sigma, a.doc.tau, a.doc.leaf_len)))
        o += len(a.doc.text)
    arrivals = staged
    gen_s = time.perf_counter() - t0
    # A warm-up pass over the whole stream (streams, generators, memory pools
    # and the first use of every kernel, the library's and torch's), then the
    # measured run on a fresh server.
    warm = serve.Server(hbm_budget=120 << 30, lanes=lanes, queries_per_doc=10_000, small_max=small_max)
    warm.run(arrivals)
    warm.close()
    srv = serve.Server(hbm_budget=120 << 30, lanes=lanes, queries_per_doc=10_000, small_max=small_max)
    rep = srv.run(arrivals)
    srv.close()
    out = rep.summary()
    out["generate_s"] = gen_s
    out["offered_mb_per_s"] = sum(len(a.doc.text) for a in arrivals) / max(duration, 1e-9) / 1e6
    out["workload"] = (f"Poisson {rate:.0f} docs/s for {duration} s ({len(arrivals)} documents), log-uniform "
                       f"{min_len >> 10} KiB - {max_len >> 20} MiB, DNA-like / text-like 50/50, "
                       f"120 GiB budget, {out['queries_per_doc']} queries per document, {lanes} lanes; texts in pinned host memory")
    return out


def run_reference(args):
    world, rank, _ = dist_setup(args)
    if rank != 0:
        return
    w = WORKLOADS[args.workload]
    text = w["gen"]()
    n = min(len(text), args.cpu_sample_mib << 20)
    import oracle
    sample = np.ascontiguousarray(text[:n])
    for _ in range(args.warmup):
        oracle.build(sample, w["tau"], w["leaf"], prune=True)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.build(sample, w["tau"], w["leaf"], prune=True)
    sec = time.perf_counter() - t0
    value = n * args.steps / sec / 1e6
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": sec * 1e3 / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u8",
        "data": "synthetic",
        "config": {"workload": args.workload, "n": n, "sigma": w["sigma"], "tau": w["tau"],
                   "leaf_len": w["leaf"], "prune": True, "sample": f"first {n >> 20} MiB"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"first {n} bytes of the {args.workload} text per step"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def scan_roofline(prof: dict, step_ms_total: float, traffic_ratio: float | None) -> dict:
    """Roofline of the window scan from the library's CUDA-event profile:
    covered bytes of the timed levels / their event time, against the
    measured HBM copy bandwidth."""
    hbm = measured_peaks().get("hbm_gbs")
    scan = prof.get("window_scan", {"launches": 0, "ms": 0.0, "bytes": 0})
    achieved = scan["bytes"] / (scan["ms"] / 1e3) / 1e9 if scan["ms"] > 0 else None
    per_launch_bytes = scan["bytes"] / max(1, scan["launches"])
    return {
        "kernel": "a level's leftmost occurrences (bounds, comparisons and the search of the open keys; "
                  "k_scan_anchor, k_hits and k_candidates on levels of blocks under 27 bytes): covered bytes "
                  "per second, most of which are settled without being read",
        "bound": "hbm",
        "achieved": achieved,
        "peak": hbm if hbm else 6800.0,
        "peak_source": "of measured (MEASURED_PEAKS.json hbm_gbs)" if hbm else "of fallback",
        "unit": "GB/s",
        "frac": (achieved / hbm) if (achieved and hbm) else None,
        "frac_of_spec": (achieved / HBM_SPEC_GBS) if achieved else None,
        "traffic": (traffic_ratio * per_launch_bytes) if traffic_ratio is not None else None,
        "alg_bytes_per_launch": per_launch_bytes,
        "launches": scan["launches"],
        "share_of_step": (scan["ms"] / step_ms_total) if step_ms_total > 0 else None,
    }


def measure_single_text(bt, torch, stream, name: str, steps: int, warmup: int) -> dict:
    """Another single-text workload (the 2 GiB DNA copies by default), timed
    the same way as the headline: device-resident input, CUDA events over
    `steps` builds after `warmup`; then end to end from pinned host memory
    with the export read back."""
    w = WORKLOADS[name]
    t0 = time.perf_counter()
    text = w["gen"]()
    gen_s = time.perf_counter() - t0
    n = len(text)
    d_text = torch.from_numpy(text).cuda()
    opts = bt.BuildOptions(prune=True, **w.get("opts", {})).to_c()[0]

    def step(src):
        return bt.bt_build_ex(src, n, w["sigma"], w["tau"], w["leaf"], opts, stream)

    for _ in range(warmup):
        bt.bt_free(step(d_text))
    torch.cuda.synchronize()
    bt.bt_profile_reset()
    bt.bt_profile_enable(True)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(steps):
        bt.bt_free(step(d_text))
    e1.record(stream)
    torch.cuda.synchronize()
    bt.bt_profile_enable(False)
    prof = bt.bt_profile_read()
    ms = e0.elapsed_time(e1)
    h = step(d_text)
    stats = bt.bt_stats(h)
    tree_bytes = bt.bt_device_bytes(h)
    bt.bt_free(h)
    del d_text
    pinned = torch.from_numpy(text).pin_memory()
    h = step(pinned)
    out = torch.empty(len(bt.bt_export(h)), dtype=torch.uint8, pin_memory=True)  # the export, read back pinned
    bt.bt_free(h)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    d2h = 0
    for _ in range(steps):
        h = step(pinned)
        d2h = bt.bt_export_into(h, out)
        bt.bt_free(h)
    torch.cuda.synchronize()
    e2e_ms = (time.perf_counter() - t0) * 1e3
    hbm = measured_peaks().get("hbm_gbs") or 6800.0
    cov = sum(s["cov"] for s in stats)
    alg = n + cov + sum(s["verify_bytes"] for s in stats) + tree_bytes
    step_ms = ms / steps
    return {"workload": name, "desc": w["desc"], "n": n, "sigma": w["sigma"], "tau": w["tau"],
            "leaf_len": w["leaf"], "build_options": w.get("opts", {}), "generate_s": gen_s,
            "value": throughput_mbs(n, steps, 1, ms), "unit": UNIT, "steps": steps, "warmup": warmup,
            "ms_per_step": step_ms, "levels": len(stats), "sum_cov_bytes": cov,
            "roofline": scan_roofline(prof, ms, None),
            "build_roofline": {"alg_bytes_per_step": alg, "achieved": alg / (step_ms / 1e3) / 1e9,
                               "peak": hbm, "unit": "GB/s", "frac": alg / (step_ms / 1e3) / 1e9 / hbm},
            "kernels_ms_per_step": {k: v["ms"] / steps for k, v in prof.items()},
            "e2e": {"value": throughput_mbs(n, steps, 1, e2e_ms), "unit": UNIT, "h2d_bytes_per_step": n,
                    "d2h_bytes_per_step": d2h}}


def run_ours(args):
    import torch

    from paper_2512_23314_gb300 import bt

    world, rank, local = dist_setup(args)
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.cuda.current_device()
    w = WORKLOADS[args.workload]
    text = w["gen"]()
    n = len(text)
    d_text = torch.from_numpy(text).cuda()
    stream = torch.cuda.current_stream()
    opts = bt.BuildOptions(prune=True, **w.get("opts", {})).to_c()[0]

    def step(src):
        h = bt.bt_build_ex(src, n, w["sigma"], w["tau"], w["leaf"], opts, stream)
        return h

    for _ in range(max(args.warmup, 0)):
        bt.bt_free(step(d_text))
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    # --- device-resident timed region ---------------------------------
    sampler = ClockSampler(dev)
    barrier()
    sampler.start()
    time.sleep(0.3)
    bt.bt_profile_reset()
    bt.bt_profile_enable(True)
    launches0 = bt.bt_launch_count()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        bt.bt_free(step(d_text))
    e1.record(stream)
    barrier()
    launches = bt.bt_launch_count() - launches0
    bt.bt_profile_enable(False)
    clocks = sampler.stop()
    prof = bt.bt_profile_read()
    ms = max_over_ranks(e0.elapsed_time(e1), world)
    value = throughput_mbs(n, args.steps, world, ms)

    # --- end to end through the C ABI with host buffers -----------------
    h = step(d_text)
    stats = bt.bt_stats(h)
    tree_bytes = bt.bt_device_bytes(h)
    blob = bt.bt_export(h)
    queries = measure_queries(bt, torch, stream, h, text) if rank == 0 else None
    bt.bt_free(h)
    compact = None
    if rank == 0:
        # Space-efficient rank/select support: no stored counters on the last
        # level (counted in the leaf text by the queries that need them).
        oc = bt.BuildOptions(prune=True, leaf_counts=True, **w.get("opts", {})).to_c()[0]
        hc = bt.bt_build_ex(d_text, n, w["sigma"], w["tau"], w["leaf"], oc, stream)
        cbytes = bt.bt_device_bytes(hc)
        compact = {"tree_device_bytes": cbytes, "default_tree_device_bytes": tree_bytes,
                   "ratio": cbytes / tree_bytes, "same_export": bt.bt_export(hc) == blob,
                   "queries": measure_queries(bt, torch, stream, hc, text)}
        bt.bt_free(hc)
    sort_variant = None
    if rank == 0 and not args.no_extras:
        sort_variant = measure_sort_variant(bt, torch, stream, d_text, n, w, blob)
    pinned = torch.from_numpy(text).pin_memory()
    out = torch.empty(len(blob), dtype=torch.uint8, pin_memory=True)  # the export, read back pinned
    barrier()
    e2 = torch.cuda.Event(enable_timing=True)
    e3 = torch.cuda.Event(enable_timing=True)
    t_host0 = time.perf_counter()
    e2.record(stream)
    d2h = 0
    for _ in range(args.steps):
        h = step(pinned)
        d2h = bt.bt_export_into(h, out)
        bt.bt_free(h)
    e3.record(stream)
    barrier()
    e2e_ms = max_over_ranks((time.perf_counter() - t_host0) * 1e3, world)
    e2e_value = throughput_mbs(n, args.steps, world, e2e_ms)

    if rank != 0:
        if world > 1:
            torch.distributed.destroy_process_group()
        return

    peaks = measured_peaks()
    hbm = peaks.get("hbm_gbs")
    roofline = scan_roofline(prof, ms, recorded_traffic("window_scan"))
    cov = sum(s["cov"] for s in stats)
    mulmods, mwork = issued_mulmods(n, stats)
    int_roof = int_roofline(bt, torch, stream, mulmods, ms / args.steps, mwork)
    vbytes = sum(s["verify_bytes"] for s in stats)
    cands = sum(s["candidates"] for s in stats)
    hits = sum(s["hits"] for s in stats)
    # The whole build against the same peak (B_alg = n + sum cov + V + S, S the tree's bytes).
    alg_build = n + cov + vbytes + tree_bytes
    build_gbs = alg_build / (ms / args.steps / 1e3) / 1e9 * world if ms > 0 else None
    t_hbm_ms = alg_build / ((hbm if hbm else 6800.0) * 1e9) * 1e3
    build_roofline = {"alg_bytes_per_step": alg_build, "achieved": build_gbs,
                      "peak": hbm if hbm else 6800.0, "unit": "GB/s",
                      "frac": (build_gbs / hbm) if (build_gbs and hbm) else None,
                      "frac_of_spec": (build_gbs / HBM_SPEC_GBS) if build_gbs else None,
                      "t_roof_hbm_ms": t_hbm_ms, "t_roof_int_ms": int_roof["t_roof_ms"],
                      "larger_roof": "int" if int_roof["t_roof_ms"] > t_hbm_ms else "hbm"}
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u8", "data": "synthetic",
        "config": {"workload": args.workload, "n": n, "sigma": w["sigma"], "tau": w["tau"],
                   "leaf_len": w["leaf"], "prune": True, "build_options": w.get("opts", {}),
                   "levels": len(stats),
                   "sum_cov_bytes": cov, "verify_bytes": vbytes, "scan_candidates": cands,
                   "scan_hits": hits,
                   "l2": "input (n bytes) larger than the 129 MB L2; no flush",
                   "parallelism": "replicas" if world > 1 else "single GPU"},
        "roofline": roofline,
        "build_roofline": build_roofline,
        "int_roofline": int_roof,
        "queries": queries,
        "leaf_counts": compact,
        "sort_scan": sort_variant,
        "kernels_ms_per_step": {k: v["ms"] / args.steps for k, v in prof.items()},
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": n,
                "d2h_bytes_per_step": d2h},
        "gpu_launches": launches,
        "clocks": clocks,
    }
    if world == 1 and not args.no_extras:
        # The headline is the 256 MiB versioned text (the workload the metric is
        # quoted on); the 2 GiB DNA copies, the batched workload and the serving
        # loop are measured beside it.
        line["configs"] = {"dna_genome_2GiB": measure_single_text(bt, torch, stream, "dna_genome_2GiB",
                                                                  steps=3, warmup=2)}
        line["batch"] = measure_batch(args.batch_docs, max_len=args.batch_max_mib << 20)
        line["serve"] = measure_serve()
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(text, w, args.cpu_sample_mib)
        line["cpu_mt_baseline"] = cpu_mt_baseline(text, w, args.cpu_mt_sample_mib)
    print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


def main():
    args = parse_args()
    if args.summarize_launches:
        summarize_launches(args.summarize_launches, args.builds)
    elif args.summarize_traffic:
        summarize_traffic(*args.summarize_traffic, args.builds)
    elif args.batch_only:
        import torch
        torch.cuda.set_device(0)
        print(json.dumps(measure_batch(args.batch_docs, max_len=args.batch_max_mib << 20)), flush=True)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
