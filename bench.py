#!/usr/bin/env python
"""Throughput of exact triangle counting (forward algorithm) on GB300.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--workload rmat24|rmat20|rgg4m|er16k]

One step = the whole path (validation, cleaning, degree-ordered orientation,
an LSD radix sort by owner, node array, per-list sorts that drop repeated
edges, partner groups, counting with per-vertex counts) over one
graph whose edge array is already resident in HBM.  The default workload is
the R-MAT graph of scale 24 with 180,000,000 distinct undirected edges
(a=.57, b=.19, c=.19, d=.05, seed 1004), whose per-vertex counts feed the
clustering coefficient and transitivity.  Its inputs (1.44 GB) and key
buffers (2.9 GB) are far larger than the 126 MB L2, so no flush is needed
between steps.

Printed: one JSON line on rank 0.  `value` is input pairs per second over
all ranks.  With N > 1 GPUs (torchrun) the ranks count ONE graph by default:
every rank preprocesses its own copy, counts its share of the partner groups
(tc_count_per_vertex_part) and one sum all-reduce joins the shares
(Sec. III-E, strong scaling); `--replicas` lets each rank count its own copy
instead (weak scaling).
Beside the main line: the same graph in the paper's input format (every
edge in both directions, Sec. III-A; `paper_format`), end to end through the
host-buffer call (`e2e`), the CPU oracle on a sample (`cpu_baseline`),
stand-ins of the paper's synthetic Table 1 graphs timed as the paper times
them (`paper_table1`) and the 4096-graph batch (`batched`).
`--impl reference` times the CPU oracle (the paper's own baseline is a
single-threaded CPU forward algorithm, Sec. IV) on a bounded sample of the
same workload, on the host cores.
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

METRIC = "input edges/s"
UNIT = "edges/s"
CPU_SAMPLE_PAIRS = 24_000_000      # cpu_baseline: first pairs of the workload
REF_SAMPLE_PAIRS = 6_000_000       # reference arm: per step
KERNEL_OF_PHASE = {"canon": "k_canon", "lists": "k_sort_lists",
                   "rank": "k_rank_keys+k_radix_pass",
                   "orient": "k_orient", "sort": "k_radix_pass", "offsets": "k_offsets",
                   "groups": "k_group_keys+k_radix_pass+k_offsets", "count": "k_count"}


def parse_args():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=10)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", choices=["ours", "reference"], default="ours")
    p.add_argument("--workload", default="rmat24")
    p.add_argument("--e2e-steps", type=int, default=3)
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--cpu-full", action="store_true",
                   help="time the CPU oracle on the WHOLE workload (rmat24: about ten "
                        "minutes on one core) instead of the bounded sample")
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--no-paper-table", action="store_true",
                   help="skip the stand-ins of the paper's synthetic Table 1 graphs (T only, "
                        "host to host, the paper's timing protocol)")
    p.add_argument("--no-paper-format", action="store_true",
                   help="skip timing the same graph in the paper's input format (every edge "
                        "in both directions, 2m pairs), checked against the main run")
    p.add_argument("--total-only", action="store_true",
                   help="time tc_count (T only) instead of tc_count_per_vertex")
    p.add_argument("--no-batched", action="store_true",
                   help="skip the 4096-graph batched vs per-graph-loop comparison")
    p.add_argument("--batch-graphs", type=int, default=4096)
    p.add_argument("--serve-graphs", type=int, default=2048,
                   help="requests per arrival rate in the serving run (0: skip it)")
    p.add_argument("--replicas", action="store_true",
                   help="with several GPUs, let each rank count its own replica of the graph "
                        "(weak scaling).  Default: all ranks count ONE graph, each its share "
                        "of the partner groups, joined by one sum all-reduce (Sec. III-E; "
                        "strong scaling)")
    return p.parse_args()


def log(*a):
    print(*a, file=sys.stderr, flush=True)


# ---------------------------------------------------------------- distributed
def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    pg = None
    if world > 1:
        import torch.distributed as dist

        backend = "nccl" if args.impl == "ours" else "gloo"
        dist.init_process_group(backend=backend)
        pg = dist
    return world, rank, local, pg


def barrier(pg, dev=None):
    if pg is not None:
        if dev is not None:
            pg.barrier(device_ids=[dev])
        else:
            pg.barrier()


def step_stats(ms: list) -> dict:
    """Mean, standard deviation, median and range of per-step times (this
    rank's), as the paper reports its repeats (Sec. IV: mean of five runs,
    deviation within 5%)."""
    return {"mean": round(statistics.mean(ms), 4), "std": round(statistics.pstdev(ms), 4),
            "median": round(statistics.median(ms), 4), "min": round(min(ms), 4),
            "max": round(max(ms), 4), "steps": len(ms)}


def gather_over_ranks(pg, values, dev=None) -> list:
    """Every rank's list of integers (same length on all ranks), on every
    rank; [values] alone without a process group."""
    if pg is None:
        return [list(values)]
    import torch

    t = torch.tensor([int(v) for v in values], dtype=torch.int64,
                     device="cuda" if dev is not None else "cpu")
    parts = [torch.zeros_like(t) for _ in range(pg.get_world_size())]
    pg.all_gather(parts, t)
    return [[int(x) for x in p.tolist()] for p in parts]


def max_over_ranks(pg, x: float, dev=None) -> float:
    if pg is None:
        return x
    import torch

    t = torch.tensor([x], dtype=torch.float64, device="cuda" if dev is not None else "cpu")
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    return float(t.item())


# ---------------------------------------------------------------- clocks
class ClockSampler:
    """nvidia-smi samples of this GPU's clocks and throttle reasons."""

    FIELDS = ("uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid: str | None):
        self.uuid = uuid
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, ValueError):
            self.proc = None

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) < 8:
                    continue
                if self.uuid and parts[0] != self.uuid:
                    continue
                rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[4 + i] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


def gpu_uuid(dev) -> str | None:
    try:
        import torch

        u = str(torch.cuda.get_device_properties(dev).uuid)
        return u if u.startswith("GPU-") else "GPU-" + u
    except Exception:
        return None


# ---------------------------------------------------------------- roofline
def measured_peaks() -> dict:
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return json.load(f)
    return {}


def kernel_source_hash() -> str:
    h = hashlib.sha256()
    for name in ("preprocess.cu", "direct.cu", "group.cu", "bits.cu", "count.cu", "hub.cu",
                 "tc_common.cuh"):
        with open(os.path.join(ROOT, "paper_1503_00576_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def committed_traffic(kernel: str, workload: str):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    on the current kernel sources; else None."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(path):
        return None
    with open(path) as f:
        data = json.load(f)
    rec = data.get(workload, {}).get(kernel)
    if not rec or rec.get("source_hash") != kernel_source_hash():
        return None
    return rec.get("dram_bytes_per_launch")


def roofline(prof: dict, steps: int, m_in: int, m: int, n: int, workload: str,
             work: dict, total_only: bool = False) -> dict:
    """Dominant kernel by device time; achieved = algorithmic bytes per
    launch / average launch duration (CUDA events on the launch stream).

    The counting phase is one unit: the dense block's product, the bitmap
    intersections, the partners' streams and the two kernels that count by
    hashing share one work list and run back to back once per step, followed by
    the small gather of t[] to vertex ids.  Its algorithmic bytes are what the
    timed call's intersections read, counted by tc_debug_run_work over the groups
    and streams of that very call: each partner group's hashed list once
    (inserts) and, per partner, the part of the list streamed through it
    (lookups), 4 bytes each, and 512 bytes per partner intersected by bitmaps --
    plus the partner ids (4 each; without the count, 4m), both offset arrays
    (8(n+1)) and, per vertex, t[] in rank space written, gathered and written
    again (28n).  Most of it is served by L2, so `frac` compares a rate of bytes
    used with the HBM peak; it is not DRAM traffic (see `traffic`)."""
    b = max(1, (max(n, 2) - 1).bit_length())
    passes2 = (b + 7) // 8
    per_kernel = {}
    for phase, (ms, launches) in prof.items():
        k = KERNEL_OF_PHASE[phase]
        a = per_kernel.setdefault(k, [0.0, 0])
        a[0] += ms
        a[1] += launches
    kernel = max(per_kernel, key=lambda k: per_kernel[k][0])
    ms_total, launches = per_kernel[kernel]
    extra = {}
    if kernel == "k_count":
        kernel = "k_count+k_count_big"
        units = steps
        pairs, partners = work.get("bitmap_pairs", 0), work.get("partners", m)
        lists = 4 * (work["lookups"] + work["inserts"]) + 512 * pairs
        bytes_per_launch = lists + 4 * partners + 8 * (n + 1) + (0 if total_only else 28 * n)
        how = ("one counting phase: 4 B per list element read by the hash intersections "
               "(lookups %d + inserts %d) + 512 B per bitmap intersection (%d) + partner ids "
               "(%d) + offsets 8(n+1)%s"
               % (work["lookups"], work["inserts"], pairs, partners,
                  "" if total_only else " + t[] 28n"))
        t = ms_total / 1e3 / units
        extra = {"kernels_timed": "k_hub_zero, k_hub_scatter, k_hub_gemm, k_hub_finish, "
                                  "k_count_bits, k_stream_desc, k_count_big, k_count, "
                                  "k_gather_counts (those that the call launches)",
                 "merge_equivalent_gbs": round(4 * work["merge_work"] / t / 1e9, 1),
                 "merge_work_W": work["merge_work"],
                 "compulsory_gbs": round((4 * m + 4 * (n + 1) + (0 if total_only else 8 * n))
                                         / t / 1e9, 1)}
    elif kernel == "k_radix_pass":
        units = launches
        total = (passes2 - 1) * 16 * m_in + 12 * m_in
        bytes_per_launch = total / passes2
        how = ("sort by owner: 8-byte key read + 8-byte key write per key per pass (the last "
               "pass writes 4 + 4 bytes)")
    else:
        units = launches
        bytes_per_launch = 16 * m_in
        how = "16 bytes per input pair"
    per_launch_s = ms_total / 1e3 / max(units, 1)
    achieved = bytes_per_launch / per_launch_s / 1e9
    peaks = measured_peaks()
    peak = peaks.get("hbm_gbs")
    src = "measured"
    if not peak:
        peak, src = 6800.0, "fallback"
    return {"bound": "hbm", "kernel": kernel, "achieved": round(achieved, 1), "peak": peak,
            "unit": "GB/s", "frac": round(achieved / peak, 4), "peak_source": src,
            "traffic": committed_traffic(kernel, workload),
            "algorithmic_bytes_per_launch": int(bytes_per_launch), "bytes_rule": how,
            "launches_timed": units, "ms_per_launch": round(per_launch_s * 1e3, 4), **extra}


# ---------------------------------------------------------------- CPU oracle timing
def time_oracle(src, dst, n, pairs: int) -> tuple[float, int]:
    import oracle

    pairs = min(pairs, len(src))
    t0 = time.perf_counter()
    oracle.forward(src[:pairs], dst[:pairs], n)
    return time.perf_counter() - t0, pairs


# ---------------------------------------------------------------- batched
def stored_batch_totals(count: int):
    """The CPU oracle's per-graph totals of graph_batch(count, 1005), written
    by tests/golden/make_batch_golden.py, or None for another batch."""
    import numpy as np

    path = os.path.join(ROOT, "tests", "golden", "batch4096.json")
    if not os.path.exists(path):
        return None
    with open(path) as f:
        gold = json.load(f)
    if gold["count"] != count or gold["seed"] != 1005:
        return None
    return np.array(gold["T"], np.uint64)


def run_batched(args, tc, rank: int = 0, world: int = 1, pg=None, dev=None) -> dict:
    """Graphs/s of the persistent CUDA-graph batch engines (autotuned) against
    the per-graph launch loop, on the same device-resident graphs; the
    per-graph counts must be identical.  With several ranks each one counts
    the graphs dealt to it (batching.deal_graphs, by size), whole and alone:
    no collective on the data path; every rank checks its own totals, one
    all-gather joins the verdicts, and the times are the maximum over the
    ranks."""
    import numpy as np
    import torch

    import graphgen
    from paper_1503_00576_gb300 import autotune, batching

    t0 = time.time()
    G_all = args.batch_graphs
    mine = None
    if world > 1:
        _, m_all, _, _ = graphgen.batch_params(G_all, 1005)
        mine = batching.deal_graphs(np.concatenate([[0], np.cumsum(m_all)]), world)[rank]
        gb = graphgen.graph_batch(G_all, 1005, only=mine,
                                  threads=max(1, (os.cpu_count() or 4) // world))
    else:
        gb = graphgen.graph_batch(G_all, 1005)
    gen_s = time.time() - t0
    G = len(gb)
    m_total = int(gb.edge_offsets[-1])
    s = torch.from_numpy(gb.src).cuda()
    d = torch.from_numpy(gb.dst).cuda()
    eo, vn = gb.edge_offsets, gb.vertex_counts
    cap = batching.Capacity()
    log("batched: %d graphs, %d pairs generated in %.1fs" % (G, m_total, gen_s))

    # per-graph launch loop (one warm pass over a prefix first)
    batching.count_plain(s, d, eo[:65], vn[:64])
    torch.cuda.synchronize()
    barrier(pg, dev)
    t0 = time.perf_counter()
    plain = batching.count_plain(s, d, eo, vn)
    torch.cuda.synchronize()
    plain_s = max_over_ranks(pg, time.perf_counter() - t0, dev)

    t0 = time.time()
    tuned = autotune.tune_batches(s, d, eo, vn, cap)
    tune_s = time.time() - t0
    with batching.BatchCounter(cap, tuning=tuned["tuning"]) as bc:
        ref = bc.count(s, d, eo, vn)  # warm
        times = []
        for _ in range(2):
            torch.cuda.synchronize()
            barrier(pg, dev)
            t0 = time.perf_counter()
            got = bc.count(s, d, eo, vn)
            torch.cuda.synchronize()
            times.append(max_over_ranks(pg, time.perf_counter() - t0, dev))
            assert np.array_equal(got, ref)
    batched_s = min(times)
    exact = bool(np.array_equal(ref, plain))
    oracle_identical = None
    gold = stored_batch_totals(G_all)
    if gold is not None:
        if mine is not None:
            gold = gold[mine]
        oracle_identical = bool(np.array_equal(ref, gold) and np.array_equal(plain, gold))
    # every rank's verdict, and the whole batch's triangles
    parts = gather_over_ranks(pg, [exact, bool(oracle_identical), int(ref.sum())], dev)
    exact = all(p[0] for p in parts)
    if gold is not None:
        oracle_identical = all(p[1] for p in parts)
    tri = sum(p[2] for p in parts)
    plan = batching.plan_subbatches(eo, vn, cap)
    del s, d
    served = None
    if args.serve_graphs > 0 and world == 1:
        torch.cuda.empty_cache()
        served = run_served(gb, ref, min(args.serve_graphs, G), G / plain_s, tuned["tuning"])
    if world > 1:
        m_total = int(graphgen.batch_params(G_all, 1005)[1].sum())
    return {"graphs": G_all, "pairs": m_total, "triangles": tri,
            "graphs_per_s": G_all / batched_s, "edges_per_s": m_total / batched_s,
            "plain_graphs_per_s": G_all / plain_s, "plain_edges_per_s": m_total / plain_s,
            "ranks": world, "graphs_per_rank": G if world == 1 else "dealt by size",
            "speedup_vs_plain": plain_s / batched_s, "counts_identical": exact,
            "oracle_identical": oracle_identical,
            "oracle_totals": "tests/golden/batch4096.json (CPU oracle, one graph per core)"
                             if gold is not None else None,
            "batched_s": batched_s, "plain_s": plain_s, "subbatches": len(plan),
            "engines": 2, "capacity": {"pairs": cap.pairs, "vertices": cap.vertices,
                                        "graphs": cap.graphs},
            "tuning": tuned["tuning"], "tuning_cached": tuned["cached"],
            "autotune_s": round(tune_s, 1), "autotune_ms": tuned["ms"], "served": served,
            "workload": "4096 graphs: half Erdos-Renyi, half R-MAT (.57,.19,.19), n "
                        "log-uniform in [2^8, 2^18], mean degree uniform in [4, 64], "
                        "seed 1005; inputs resident in HBM; wall clock, device synchronised"}


def run_served(gb, want, G: int, plain_rate: float, tuning) -> dict:
    """Continuous-batching server under seeded Poisson arrivals of the first
    G graphs of the batch, at 0.5x, 1x and 2x the per-graph loop's rate.
    Requests come from page-locked host memory (the copy to the device is
    part of each request's latency); every result must equal the batched
    count of its graph."""
    import numpy as np
    import torch

    from paper_1503_00576_gb300 import batching, serve

    eo = gb.edge_offsets
    t0 = time.time()
    ps = torch.from_numpy(gb.src[:eo[G]]).pin_memory()
    pd = torch.from_numpy(gb.dst[:eo[G]]).pin_memory()
    pin_s = time.time() - t0
    reqs = [(ps[eo[g]:eo[g + 1]], pd[eo[g]:eo[g + 1]], int(gb.vertex_counts[g]))
            for g in range(G)]
    cap = batching.Capacity(pairs=1 << 26, vertices=1 << 23, graphs=1024)
    out = {"requests_per_rate": G, "pairs": int(eo[G]), "plain_graphs_per_s": plain_rate,
           "engines": 2, "capacity": {"pairs": cap.pairs, "vertices": cap.vertices,
                                      "graphs": cap.graphs},
           "tuning": tuning, "pin_s": round(pin_s, 2), "rates": []}
    exact = True
    with serve.Server(cap, engines=2, tuning=tuning) as srv:
        for f in [srv.submit(*r) for r in reqs[:64]]:  # warm
            f.result()
        srv.drain()
        srv.stats(reset=True)
        for mult in (0.5, 1.0, 2.0):
            rate = mult * plain_rate
            futs = serve.poisson_stream(srv, reqs, rate, seed=1005)
            srv.drain(timeout=600)
            got = np.array([f.result() for f in futs], np.uint64)
            ok = bool(np.array_equal(got, want[:G]))
            exact &= ok
            st = srv.stats(reset=True)
            st.update({"offered_x_plain": mult, "offered_graphs_per_s": rate,
                       "edges_per_s": int(eo[G]) / st["span_s"], "counts_identical": ok})
            out["rates"].append({k: (round(v, 4) if isinstance(v, float) else v)
                                 for k, v in st.items()})
            log("served %.1fx: %s" % (mult, out["rates"][-1]))
    out["counts_identical"] = exact
    out["workload"] = ("first %d graphs of the 4096-graph batch, Poisson arrivals (seed 1005) "
                       "from page-locked host memory; latency = submit to result" % G)
    return out


# ---------------------------------------------------------------- arms
# The synthetic rows of the paper's Table 1: row, input, the row's edge
# entries (every edge listed twice), triangles, CPU ms and GTX 980 ms.  The
# inputs are stand-ins of the same family and size: R-MAT with the Graph500
# parameters drawn until half the row's edge entries are distinct edges
# (the row's Kronecker graphs are not available), and the Barabasi-Albert
# and Watts-Strogatz generators at the rows' sizes.
PAPER_TABLE1 = [
    ("Kronecker 16", ("rmat", 16), 5e6, 119e6, 2810, 82),
    ("Kronecker 17", ("rmat", 17), 10e6, 288e6, 6957, 219),
    ("Kronecker 18", ("rmat", 18), 21e6, 688e6, 17808, 558),
    ("Kronecker 19", ("rmat", 19), 44e6, 1626e6, 45947, 1443),
    ("Kronecker 20", ("rmat", 20), 89e6, 3804e6, 116811, 3942),
    ("Kronecker 21", ("rmat", 21), 182e6, 8816e6, 297426, 12009),
    ("Barabasi-Albert", ("ba200k",), 20e6, 3e6, 5508, 155),
    ("Watts-Strogatz", ("ws1m",), 50e6, 219e6, 9627, 324),
]


def paper_table_input(spec, edges):
    import graphgen

    if spec[0] == "rmat":
        scale = spec[1]
        src, dst = graphgen.rmat_distinct(scale, int(edges // 2), 1100 + scale)
        return src, dst, 1 << scale
    return graphgen.workload(spec[0])


def run_paper_table(tc, rows=PAPER_TABLE1, repeats: int = 5) -> list:
    """T only, as the paper counts, on stand-ins of its synthetic graphs.  Its
    protocol (Sec. IV): wall clock from the inputs in host memory to the
    total back on the host, after a warm-up, mean of five runs; here through
    tc_count_host with page-locked buffers.  The device-resident time (CUDA
    events, tc_count) is given beside it.  Context only: other graphs of the
    same families and sizes, other hardware."""
    import torch

    out = []
    stream = torch.cuda.current_stream()
    for name, spec, edges, tri, cpu_ms, gtx_ms in rows:
        src, dst, n = paper_table_input(spec, edges)
        hs = torch.from_numpy(src).pin_memory()
        hd = torch.from_numpy(dst).pin_memory()
        T = tc.tc_count_host(hs, hd, n)  # warm-up
        wall = []
        for _ in range(repeats):
            torch.cuda.synchronize()
            a = time.perf_counter()
            Th = tc.tc_count_host(hs, hd, n)
            wall.append(time.perf_counter() - a)
            assert Th == T
        ds, dd = hs.cuda(), hd.cuda()
        assert tc.tc_count(ds, dd, n, stream=stream) == T
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        for _ in range(repeats):
            tc.tc_count(ds, dd, n, stream=stream)
        ev1.record(stream)
        torch.cuda.synchronize()
        ms_dev = ev0.elapsed_time(ev1) / repeats
        ms = statistics.mean(wall) * 1e3
        out.append({"graph": name, "input": graphgen_name(spec, edges), "n": int(n),
                    "pairs": int(len(src)), "triangles": int(T),
                    "ms_host_to_host": round(ms, 3),
                    "ms_host_to_host_std": round(statistics.pstdev(wall) * 1e3, 3),
                    "ms_device_resident": round(ms_dev, 3),
                    "paper": {"edge_entries": edges, "triangles": tri, "cpu_ms": cpu_ms,
                              "gtx980_ms": gtx_ms}})
        del hs, hd, ds, dd
        torch.cuda.empty_cache()
    return out


def graphgen_name(spec, edges) -> str:
    if spec[0] == "rmat":
        return ("R-MAT scale %d (a,b,c = .57,.19,.19), draws until %d distinct edges, seed %d"
                % (spec[1], int(edges // 2), 1100 + spec[1]))
    import graphgen

    return graphgen.WORKLOADS[spec[0]][0]


def run_paper_format(steps: int, tc, s, d, n: int, m: int, T: int, t_ref, deg_ref,
                     stream) -> dict:
    """The graph in the paper's input format (Sec. III-A): every edge listed in
    both directions, 2m pairs.  Each key then comes twice, so the degrees
    count every edge twice (the order stays the same) and the list sort drops
    one copy of every edge; the counts must equal the main run's."""
    import torch

    s2 = torch.cat([s, d])
    d2 = torch.cat([d, s])
    t2 = torch.empty_like(t_ref)
    deg2 = torch.empty_like(deg_ref)

    def step():
        return tc.tc_count_per_vertex(s2, d2, n, stream=stream, t_out=t2, deg_out=deg2)[0]

    for _ in range(3):
        Tp = step()
    torch.cuda.synchronize()
    identical = Tp == T and bool(torch.equal(t2, t_ref)) and bool(torch.equal(deg2, deg_ref))
    assert identical, "the paper's input format changed a count"
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(steps):
        step()
    ev1.record(stream)
    torch.cuda.synchronize()
    dt = ev0.elapsed_time(ev1) / 1e3 / steps
    pairs = int(s2.numel())
    del s2, d2, t2, deg2
    torch.cuda.empty_cache()
    return {"input": "each edge of the workload twice: the pairs, then the same pairs "
                     "reversed", "pairs": pairs, "edges": m, "steps": steps,
            "ms_per_step": dt * 1e3, "pairs_per_s": pairs / dt, "edges_per_s": m / dt,
            "identical_to_main_run": identical}


def run_reference(args, world, rank, pg):
    import graphgen

    if rank != 0:
        return
    src, dst, n = graphgen.workload(args.workload)
    times = []
    for i in range(args.warmup + args.steps):
        dt, pairs = time_oracle(src, dst, n, REF_SAMPLE_PAIRS)
        if i >= args.warmup:
            times.append(dt)
    mean = statistics.mean(times)
    value = pairs / mean
    sample = "first %d pairs of the %s edge array per step (oracle: single-threaded C " \
             "forward algorithm)" % (pairs, args.workload)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": mean * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "int64", "data": "synthetic",
            "config": {"workload": graphgen.WORKLOADS[args.workload][0], "n": n,
                       "m_in": int(len(src)), "sample_pairs_per_step": pairs,
                       "sample": "each step counts only the first %d of the %d pairs"
                                 % (pairs, len(src))},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(args, world, rank, local, pg):
    import numpy as np
    import torch

    import graphgen
    import paper_1503_00576_gb300 as tc

    torch.cuda.set_device(local)
    dev = local
    tc.load_library()
    t0 = time.time()
    src, dst, n = graphgen.workload(args.workload)
    log("rank %d: generated %s (%d pairs) in %.1fs" % (rank, args.workload, len(src),
                                                      time.time() - t0))
    m_in = len(src)
    s = torch.from_numpy(src).cuda()
    d = torch.from_numpy(dst).cuda()
    t_out = torch.empty(n, dtype=torch.int64, device="cuda")
    deg_out = torch.empty(n, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream()

    sharded = world > 1 and not args.replicas
    if sharded:
        from paper_1503_00576_gb300.shard import count_sharded

        if args.total_only:
            def step():
                return count_sharded(s, d, n, stream=stream)
        else:
            def step():
                return count_sharded(s, d, n, per_vertex=True, stream=stream)[0]
    elif args.total_only:
        def step():
            return tc.tc_count(s, d, n, stream=stream)
    else:
        def step():
            return tc.tc_count_per_vertex(s, d, n, stream=stream, t_out=t_out,
                                          deg_out=deg_out)[0]

    for _ in range(max(args.warmup, 3)):
        T = step()
    torch.cuda.synchronize()
    if args.total_only:
        tc.tc_count_per_vertex(s, d, n, stream=stream, t_out=t_out, deg_out=deg_out)
    m = int((deg_out.to(torch.int64).sum() // 2).item())
    # untimed: the work by whole lists, and what the timed call's kernels do
    # (a share is dealt by whole lists)
    work = tc.tc_count_work(s, d, n)
    assert work["edges"] == m and work["triangles"] == T
    run = work if sharded else tc.tc_debug_run_work(s, d, n, not args.total_only)
    assert run["triangles"] == T

    clocks = ClockSampler(gpu_uuid(dev))
    tc.tc_profile_read(reset=True)
    tc.tc_profile_enable(True)
    launches0 = tc.tc_launch_count()
    clocks.start()
    time.sleep(0.4)  # let the sampler take a first reading
    barrier(pg, dev)
    torch.cuda.synchronize()
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    evs[0].record(stream)
    for i in range(args.steps):
        T2 = step()
        evs[i + 1].record(stream)
    torch.cuda.synchronize()
    barrier(pg, dev)
    clk = clocks.stop()
    launches = tc.tc_launch_count() - launches0
    tc.tc_profile_enable(False)
    prof = tc.tc_profile_read(reset=True)
    assert T2 == T, "count changed between steps"
    elapsed = evs[0].elapsed_time(evs[-1]) / 1e3
    elapsed = max_over_ranks(pg, elapsed, dev)
    step_ms = step_stats([evs[i].elapsed_time(evs[i + 1]) for i in range(args.steps)])
    ms_per_step = elapsed / args.steps * 1e3
    # replicas: every rank counted its own copy; shards: all ranks one graph
    value = (1 if sharded else world) * m_in * args.steps / elapsed

    # end to end through the host-buffer entry point, pinned buffers
    e2e = None
    if not args.no_e2e and not sharded:  # the host-buffer call counts whole graphs
        hs = torch.from_numpy(src).pin_memory()
        hd = torch.from_numpy(dst).pin_memory()
        ht = torch.empty(n, dtype=torch.int64).pin_memory()
        hdeg = torch.empty(n, dtype=torch.int32).pin_memory()

        def host_step():
            if args.total_only:
                return tc.tc_count_host(hs, hd, n)
            return tc.tc_count_per_vertex_host(hs, hd, n, t_out=ht, deg_out=hdeg)[0]

        host_step()  # warm
        barrier(pg, dev)
        times = []
        for _ in range(args.e2e_steps):
            torch.cuda.synchronize()
            a = time.perf_counter()
            Te = host_step()
            times.append(time.perf_counter() - a)
            assert Te == T
        e2e_s = max_over_ranks(pg, statistics.mean(times), dev)
        e2e = {"value": world * m_in / e2e_s, "unit": UNIT, "h2d_bytes_per_step": 8 * m_in,
               "d2h_bytes_per_step": (0 if args.total_only else 12 * n) + 128,
               "ms_per_step": e2e_s * 1e3,
               "api": ("tc_count_host" if args.total_only else "tc_count_per_vertex_host")
                      + " (pinned host buffers)"}

    # the 4096-graph batch: every rank counts the graphs dealt to it
    batched = None
    if not args.no_batched:
        batched = run_batched(args, tc, rank, world, pg, dev)
    if rank != 0:
        return
    cpu = None
    if not args.no_cpu_baseline and world == 1:
        pairs_wanted = m_in if args.cpu_full else CPU_SAMPLE_PAIRS
        dt, pairs = time_oracle(src, dst, n, pairs_wanted)
        if pairs == m_in:
            sample = ("the whole %s edge array (%d pairs), single-threaded C oracle, %.1f s"
                      % (args.workload, pairs, dt))
        else:
            sample = ("first %d of the %d pairs of the %s edge array, single-threaded C "
                      "oracle, %.1f s.  A bounded sample: the pairs are in random draw order, "
                      "so this is a uniform edge sample -- a sparser graph with less merge "
                      "work per edge than the whole, on which the oracle runs several times "
                      "slower per edge (bench.py --cpu-full times the whole graph)"
                      % (pairs, m_in, args.workload, dt))
        cpu = {"value": pairs / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
               "sample": sample, "seconds": round(dt, 2)}
        if pairs < m_in and args.workload == "rmat24":
            # the whole graph takes the oracle about six minutes, too long for
            # the default run: its committed measurement rides along, marked
            # as such (profiles/cpu_oracle_rmat24.md; bench.py --cpu-full)
            cpu["whole_graph_measured_earlier"] = {
                "value": 4.87e5, "unit": UNIT, "seconds": 369.6, "cores": 1,
                "source": "profiles/cpu_oracle_rmat24.md (bench.py --cpu-full on the GB300 "
                          "host, the same oracle)"}
    paper_format = None
    if not args.no_paper_format and world == 1:
        paper_format = run_paper_format(args.steps, tc, s, d, n, m, T, t_out, deg_out, stream)
    paper_table = None
    if not args.no_paper_table and world == 1:
        paper_table = run_paper_table(tc)
    steps_ms = {k: round(v[0] / args.steps, 4) for k, v in prof.items()}
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": ms_per_step, "higher_is_better": True,
        "scaling": "strong" if sharded else "weak", "vs_baseline": None, "dtype": "int64",
        "data": "synthetic",
        "config": {"workload": graphgen.WORKLOADS[args.workload][0], "n": n, "m_in": m_in,
                   "m_distinct": m, "triangles": T,
                   "outputs": "T (uint64)" if args.total_only
                              else "T (uint64), t[n] (int64), deg[n] (int32)",
                   "l2": "no flush: inputs %.2f GB and key buffers %.2f GB exceed L2"
                         % (8 * m_in / 1e9, 16 * m_in / 1e9),
                   "parallelism": ("shards%d" % world if sharded else "replicas")
                                  if world > 1 else "single"},
        "roofline": roofline(prof, args.steps, m_in, m, n, args.workload,
                             {**work, **run}, args.total_only),
        "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": launches, "clocks": clk,
        "step_ms": step_ms, "phase_ms_per_step": steps_ms, "batched": batched,
        "paper_format": paper_format,
        "paper_table1": paper_table,
        "counting_work": {"lookups": run["lookups"], "inserts": run["inserts"],
                          "partners": run.get("partners", m),
                          "bitmap_pairs": run.get("bitmap_pairs", 0),
                          "dense_hub_vertices": run["dense_vertices"],
                          "dense_hub_triangles": run["dense_triangles"],
                          "max_out_degree": work["max_out_degree"],
                          "merge_work_W": work["merge_work"],
                          "by_whole_lists": {
                              "lookups": work["lookups"], "inserts": work["inserts"],
                              "hub_lookup_share": {str(k): round(v / max(work["lookups"], 1), 4)
                                                   for k, v in work["hub_lookups"].items()}}},
    }
    print(json.dumps(line), flush=True)


def main():
    args = parse_args()
    world, rank, local, pg = dist_setup(args)
    try:
        if args.impl == "reference":
            run_reference(args, world, rank, pg)
        else:
            run_ours(args, world, rank, local, pg)
    finally:
        if pg is not None:
            pg.destroy_process_group()


if __name__ == "__main__":
    main()
