#!/usr/bin/env python
"""Benchmark: words/s evaluated and splatted at depth d, with the image IoU
and the largest word-value error against the FP64 oracle.

Workload (the headline): the near-cusp quasi-Fuchsian group ta = tb =
1.91 + 0.05i (Grandma's recipe), all 4,649,045,868 reduced words of length 20,
8192 x 8192 uint32 hit image over [-2, 2]^2, in FP64, the precision of the
paper's renderer.  One step = one full kl_render call: image and counter
clearing, the prefix and suffix tables and the per-word render kernel.  The
same line carries the mixed-precision renders of this job and of the gasket
at length 18 (4096^2) as secondary keys, each with its own IoU and error.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Rank 0 prints one JSON line (the whole record goes to stderr: print_line).
With N > 1 (torchrun, one process per GPU) the job is sharded: rank k renders
shard k of N (kl_params.shard_index / shard_count, a partition of the words by
prefix slot) into its own image, and one reduce sums the uint32 images and the
counters onto rank 0 inside the timed region (strong scaling: value = the
job's words / the slowest rank's time).  The oracle legs (CPU baseline and
accuracy) run at N = 1 only.
"""
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
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import klsynth  # noqa: E402

METRIC = "words/sec evaluated+splatted at depth d; image IoU and max |\u0394z| vs FP64 oracle"
FP32_OPS_PER_WORD = 12    # FP32 operations of the mixed per-word map: w = v + gamma (2),
                          # |w|^2 (2), M w (4), M w / |w|^2 + alpha (2), the two floors (2)
FP64_OPS_PER_WORD = 13    # FP64 operations of the plain per-word map: w = v + gamma (2),
                          # |w|^2 (2), reciprocal refinement (3), M w (4), final FMAs (2)
DF64_OPS_PER_WORD = 117   # FP32 operations of the double-float per-word map: w = v + gamma
                          # (2 double-float sums, 11 each), |w|^2 (16), the reciprocal's Newton
                          # step (7), the two numerators (dot products, 19 each), a + b c for
                          # the two coordinates (15 each), and the two pixel keys (2 each)
FILTER_OPS_PER_WORD = 10  # FP32 operations of the certified filter that every FP64 and
                          # double-float word takes first: omega = k v + g (4), |omega|^2 (2),
                          # the two offsets from the box's center (2), the box test (2)
SMS = 152
FP32_LANES_PER_SM = 128
FP64_LANES_PER_SM = 2
SAMPLE_N = 1_000_000      # seeded index sample for the word-value errors


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-lod", action="store_true")
    ap.add_argument("--no-tiling", action="store_true")
    ap.add_argument("--no-scan", action="store_true")
    ap.add_argument("--no-maskit", action="store_true")
    ap.add_argument("--no-multiseed", action="store_true")
    ap.add_argument("--no-cull", action="store_true")
    return ap.parse_args()


def describe(c, precision: str) -> str:
    tr = f"{c.group.ta.real:g}" + (f"{c.group.ta.imag:+g}i" if c.group.ta.imag else "")
    x0, x1, y0, y1 = c.window
    return (f"grandma ta=tb={tr}, all {c.n_words:,} reduced words of length {c.depth}, "
            f"{c.width}x{c.height} uint32 hit image over [{x0:g},{x1:g}]x[{y0:g},{y1:g}], "
            f"{precision}")


def workload(world: int = 1):
    """The headline job: the near-cusp group at length 20, 8192^2, FP64."""
    c = klsynth.C3
    return c, {"workload": describe(c, "FP64"),
               "group": "grandma ta=tb=1.91+0.05i (near-cusp, quasi-Fuchsian)",
               "depth": c.depth, "words_per_step": c.n_words, "image": [c.width, c.height],
               "window": list(c.window), "precision": "fp64",
               "parallelism": ("1 GPU" if world == 1 else
                               f"{world} shards by prefix slot, uint32 image sum (NCCL reduce)"),
               "l2": "flushed between timed steps (256 MiB write)"}


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except OSError:
        return {}


class ClockSampler:
    """nvidia-smi clock / throttle sampling while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            time.sleep(0.1)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        rows = []
        try:
            with open(self.path) as f:
                for ln in f:
                    t = [x.strip() for x in ln.split(",")]
                    if len(t) >= 9:
                        rows.append(t)
        finally:
            try:
                os.unlink(self.path)
            except OSError:
                pass
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in rows for n, v in zip(names, r[5:9]) if v == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


RENDER_SOURCES = ("paper_1709_08018_gb300/csrc/kl_common.cuh",
                  "paper_1709_08018_gb300/csrc/kl_df.cuh", "paper_1709_08018_gb300/csrc/kl_cull.cuh",
                  "paper_1709_08018_gb300/csrc/kl_filter.cuh",
                  "paper_1709_08018_gb300/csrc/kl_plan.cuh",
                  "paper_1709_08018_gb300/csrc/kl_tiling.cuh",
                  "paper_1709_08018_gb300/csrc/kl_render.cu", "include/kl.h")


def code_text(src: str) -> str:
    """C/C++/CUDA source with comments removed and whitespace runs collapsed
    (string and character literals kept), so that documentation edits leave
    the hash of the code unchanged."""
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
            out.append(" ")
        else:
            out.append(c)
            i += 1
    return " ".join("".join(out).split())


def source_hash():
    """Hash of the code (comments and layout aside) of the sources the
    single-render kernels are built from."""
    h = hashlib.sha256()
    for f in RENDER_SOURCES:
        with open(os.path.join(ROOT, f), encoding="utf-8") as fh:
            h.update(code_text(fh.read()).encode())
    return h.hexdigest()[:16]


def traffic_for(kernel: str, workload_name: str):
    """DRAM bytes per launch of `kernel` on `workload_name` from the committed
    ncu summary, if it was taken on the current kernel sources; else None."""
    try:
        with open(os.path.join(ROOT, "profiles", "traffic.json")) as f:
            rec = json.load(f)
    except (OSError, ValueError):
        return None
    k = rec.get(f"{kernel}@{workload_name}")
    if not k or k.get("source_hash") != source_hash():
        return None
    return k.get("dram_bytes_per_launch")


# ---------------------------------------------------------------------------
# oracle legs (CPU): the baseline and the accuracy figures

def oracle_render(cfg, threads=None):
    """The oracle's tree-walk render of a whole workload on the host cores,
    edge words logged at the FP64 tolerance band (1e-9 in z); returns
    (render, seconds, threads)."""
    import oracle
    threads = threads or os.cpu_count() or 1
    g, s = oracle.group(cfg.group.ta, cfg.group.tb)
    sx = cfg.width / (cfg.window[1] - cfg.window[0])
    t0 = time.perf_counter()
    r = oracle.render(g, s, cfg.depth, cfg.window, cfg.width, cfg.height, threads=threads,
                      eta=1e-9 * sx, edge_cap=1 << 22)
    return r, time.perf_counter() - t0, threads


def oracle_sample(cfg):
    """The seeded index sample and its word values by the oracle's per-word
    definition (one orbit of d maps per word)."""
    import oracle
    idx = klsynth.index_sample(klsynth.SAMPLE_SEED, SAMPLE_N, cfg.depth)
    g, s = oracle.group(cfg.group.ta, cfg.group.tb)
    return idx, oracle.evaluate(g, s, cfg.depth, idx)


def cpu_baseline(cfg, rend, secs, threads):
    return {"value": cfg.n_words / secs, "unit": "words/s", "cores": threads, "kind": "oracle",
            "sample": f"the whole workload: all {cfg.n_words} words of length {cfg.depth} "
                      f"(FP64 tree walk, {threads} threads, edge words logged)",
            "seconds": secs}


def occupancy_iou(a, b) -> float:
    oa, ob = a > 0, b > 0
    union = int((oa | ob).sum())
    return 1.0 if union == 0 else int((oa & ob).sum()) / union


def image_agreement(got, ref):
    """Agreement of a GPU image (H, W uint32) with an oracle render."""
    import numpy as np
    d = got.astype(np.int64) - ref.image.astype(np.int64)
    return {"iou_vs_oracle": occupancy_iou(got, ref.image),
            "pixels_differing": int((d != 0).sum()), "l1_hit_difference": int(np.abs(d).sum()),
            "oracle_edge_words": int(ref.edge_total)}


def sample_dz(cfg, uv, z):
    """Largest |dz| / max(1, |z|) and |dz| over the sample: uv are the GPU's
    pixel coordinates (kl_eval_words), z the oracle's word values."""
    import numpy as np
    x0, x1, y0, y1 = cfg.window
    sx, sy = cfg.width / (x1 - x0), cfg.height / (y1 - y0)
    zg = (x0 + uv[:, 0] / sx) + 1j * (y1 - uv[:, 1] / sy)
    fin = np.isfinite(z) & (np.abs(z) < 1e12)
    dz = np.abs(zg[fin] - z[fin])
    return {"max_dz_rel": float((dz / np.maximum(1.0, np.abs(z[fin]))).max()),
            "max_dz_abs": float(dz.max()), "sample": f"{SAMPLE_N} indices, SplitMix64(1709)"}


def run_reference(args):
    """The CPU oracle as the reference arm (rank 0 only), on the headline
    workload: each step renders a bounded sample of it (equal-size tree-walk
    jobs), sized so that warmup + steps end in about two minutes."""
    world, rank, _ = dist_env()
    cfg, config = workload(world)
    if rank != 0:
        return
    import oracle
    g, s = oracle.group(cfg.group.ta, cfg.group.tb)
    jobs = oracle.tree_jobs(cfg.depth)
    threads = os.cpu_count() or 1
    per_job = cfg.n_words // jobs
    t0 = time.perf_counter()
    oracle.render(g, s, cfg.depth, cfg.window, cfg.width, cfg.height, threads=threads,
                  jobs=(0, threads))
    probe = (time.perf_counter() - t0) / threads
    per_step = 120.0 / max(1, args.steps + args.warmup)
    chunk = int(max(1, min(jobs, per_step / max(probe, 1e-9))))
    times = []
    for k in range(args.warmup + args.steps):
        j0 = (k * chunk) % jobs
        j1 = min(jobs, j0 + chunk)
        t0 = time.perf_counter()
        oracle.render(g, s, cfg.depth, cfg.window, cfg.width, cfg.height, threads=threads,
                      jobs=(j0, j1))
        dt = time.perf_counter() - t0
        if k >= args.warmup:
            times.append((dt, (j1 - j0) * per_job))
    secs = sum(t for t, _ in times)
    words = sum(w for _, w in times)
    value = words / secs
    sample = (f"{chunk} of {jobs} equal tree-walk jobs per step ({chunk * per_job} of "
              f"{cfg.n_words} words), FP64 oracle, {threads} threads")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "words/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1000.0 * secs / len(times), "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config,
            "cpu_baseline": {"value": value, "unit": "words/s", "cores": threads,
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": "words/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def tiling_config(kl, dev, steps: int, flush):
    """Tiling mode of the bench group: every node of the word tree, all
    lengths 1..18 (2 (3^18 - 1) = 774,840,976 words), mixed, 4096^2; one
    kl_render call per step, L2 flushed between steps."""
    import torch
    cfg = klsynth.C2
    p = kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width, cfg.height, cfg.window,
                       kl.MIXED, mode=kl.TILING)
    r = kl.Renderer(p, device=dev)
    for _ in range(3):
        r()
    K = max(3, min(steps, 20))
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(K)]
    torch.cuda.synchronize(dev)
    for k in range(K):
        flush.fill_(k & 0xFF)
        ev[k][0].record()
        r()
        ev[k][1].record()
    torch.cuda.synchronize(dev)
    ms = statistics.mean(a.elapsed_time(b) for a, b in ev)
    words = 2 * (3 ** cfg.depth - 1)
    cnt = r.counters.cpu().tolist()
    assert int(cnt[0]) + int(cnt[1]) == words
    return {"workload": "tiling mode: every node of the word tree of the gasket ta=tb=2, "
                        "lengths 1..18, 4096x4096 uint32, window [-1.5,1.5]^2, mixed",
            "words_per_step": words, "ms_per_step": ms, "words_per_s": words / (ms / 1000.0),
            "steps": K, "fp64_words": int(cnt[2])}


def scan_config(kl, dev, flush):
    """The paper's words of a general presentation (kl_render_fsa): the strings
    of 14 letters that the indexed Cayley table of the gasket group keeps out of
    the unpruned 4-ary tree, FP64, against the reduced-index render of the
    same words (FP64 and mixed)."""
    import torch
    d, W = 14, 4096
    window = (-1.5, 1.5, -1.5, 1.5)
    # the indexed Cayley table of the once-punctured torus (Sec. "Cayley
    # Multiplication Tables"): states and symbols I, a, b, A, B = 0..4
    table = [[0, 1, 2, 3, 4], [1, 1, 2, 0, 4], [2, 1, 2, 3, 0], [3, 0, 2, 3, 4], [4, 1, 0, 3, 4]]
    p = kl.params_init(klsynth.GASKET.ta, klsynth.GASKET.tb, d, W, W, window, kl.FP64)
    f = kl.fsa_from_params(table, p)
    img = torch.empty((W, W), dtype=torch.int32, device=dev)
    cnt = torch.zeros(kl.KL_N_COUNTERS, dtype=torch.int64, device=dev)

    def timed(fn, K=5):
        for _ in range(2):
            fn()
        ms = []
        for k in range(K):
            flush.fill_(k & 0xFF)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            torch.cuda.synchronize(dev)
            ms.append(a.elapsed_time(b))
        return statistics.median(ms)
    scan_ms = timed(lambda: kl.render_fsa(f, p, img, cnt))
    kept = int(cnt[2].item())
    r64 = kl.Renderer(p, device=dev)
    reduced64_ms = timed(lambda: r64())
    pm = kl.params_init(klsynth.GASKET.ta, klsynth.GASKET.tb, d, W, W, window, kl.MIXED)
    rm = kl.Renderer(pm, device=dev)
    reduced_mixed_ms = timed(lambda: rm())
    return {"workload": "gasket ta=tb=2, the strings of 14 letters that the indexed Cayley "
                        "table keeps (walked as a tree, no other string is looked at), "
                        "FP64, 4096^2",
            "kept_words": kept, "ms": scan_ms,
            "kept_words_per_s": kept / (scan_ms / 1000.0),
            "reduced_index_fp64_ms": reduced64_ms, "reduced_index_mixed_ms": reduced_mixed_ms,
            "speedup_reduced_index_mixed_over_table": scan_ms / reduced_mixed_ms}


def maskit_config(kl, dev, flush):
    """The paper's example: Maskit's slice at mu = -0.097 + 1.838i, depth 14,
    tiling mode (every node of the tree, all lengths 1..14).  By the indexed
    Cayley table: the strings of every length k that it keeps out of 4^k
    (kl_render_fsa, FP64, one call per length); by index: the 2 (3^14 - 1)
    reduced words (kl_render, tiling mode, FP64, double-float and mixed).  One period of the limit set, 4096^2."""
    import torch
    d, W = 14, 4096
    window = (-1.0, 1.0, -0.08, 1.92)
    table = [[0, 1, 2, 3, 4], [1, 1, 2, 0, 4], [2, 1, 2, 3, 0], [3, 0, 2, 3, 4], [4, 1, 0, 3, 4]]
    gens, seeds8 = kl.maskit(-0.097 + 1.838j)
    img = torch.empty((W, W), dtype=torch.int32, device=dev)
    cnt = torch.zeros(kl.KL_N_COUNTERS, dtype=torch.int64, device=dev)

    def timed(fn, K=5):
        for _ in range(2):
            fn()
        ms = []
        for k in range(K):
            flush.fill_(k & 0xFF)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            torch.cuda.synchronize(dev)
            ms.append(a.elapsed_time(b))
        return statistics.median(ms)

    pk = [kl.params_group(gens, seeds8, k, W, W, window, kl.FP64, accumulate=int(k > 1))
          for k in range(1, d + 1)]
    f = kl.fsa_from_params(table, pk[0])

    def all_lengths():
        for p in pk:
            kl.render_fsa(f, p, img, cnt)
    scan_ms = timed(all_lengths)
    scan_img = img.clone()
    nodes = 2 * (3 ** d - 1)
    assert int(cnt[0].item()) + int(cnt[1].item()) == nodes
    out = {"workload": "Maskit mu = -0.097+1.838i, depth 14, tiling mode (all lengths 1..14), "
                       "window [-1,1]x[-0.08,1.92], 4096^2",
           "nodes": nodes, "by_table_fp64_ms": scan_ms}
    for name, prec in (("fp64", kl.FP64), ("df64", kl.DF64), ("mixed", kl.MIXED)):
        p = kl.params_group(gens, seeds8, d, W, W, window, prec, mode=kl.TILING)
        r = kl.Renderer(p, device=dev)
        out[f"indexed_{name}_ms"] = timed(lambda: r())
        if name in ("fp64", "df64"):
            diff = int((r.image.to(torch.int64) - scan_img.to(torch.int64)).abs().sum().item())
            out[f"{name}_images_differ_in_hits"] = diff
    out["speedup_indexed_fp64_over_table"] = scan_ms / out["indexed_fp64_ms"]
    out["speedup_indexed_df64_over_table"] = scan_ms / out["indexed_df64_ms"]
    out["speedup_indexed_mixed_over_table"] = scan_ms / out["indexed_mixed_ms"]
    return out


def multiseed_config(kl, dev, flush):
    """Multi-seed feeding: every reduced word of length 18 of the gasket drawn
    once per point of kl_cusp_seeds (8 points: the attracting fixed points of
    a, b, A, B and the fixed points of abAB, bABa, ABab, BabA), 4096^2, FP64
    and mixed; against the one-seed-per-letter render of the same words."""
    import torch
    c = klsynth.C2
    W = c.width
    img = torch.empty((W, W), dtype=torch.int32, device=dev)
    cnt = torch.zeros(kl.KL_N_COUNTERS, dtype=torch.int64, device=dev)

    def timed(fn, K=5):
        for _ in range(2):
            fn()
        ms = []
        for k in range(K):
            flush.fill_(k & 0xFF)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            torch.cuda.synchronize(dev)
            ms.append(a.elapsed_time(b))
        return statistics.median(ms)

    out = {"workload": "gasket ta=tb=2, length 18, 8 seed points, 4096^2, window [-1.5,1.5]^2",
           "points": 8, "words_per_render": c.n_words, "words_per_call": 8 * c.n_words}
    for name, prec in (("fp64", kl.FP64), ("df64", kl.DF64), ("mixed", kl.MIXED)):
        p = kl.params_init(c.group.ta, c.group.tb, c.depth, W, W, c.window, prec)
        s16 = kl.cusp_seeds(list(p.gens))
        pts = [complex(s16[2 * i], s16[2 * i + 1]) for i in range(8)]
        ws = torch.empty(kl.workspace_bytes(p), dtype=torch.uint8, device=dev)
        ms = timed(lambda: kl.render_multiseed(p, pts, img, cnt, ws))
        assert int(cnt[0].item()) + int(cnt[1].item()) == 8 * c.n_words
        one = kl.Renderer(p, device=dev)
        one_ms = timed(lambda: one())
        out[f"{name}_ms"] = ms
        out[f"{name}_words_per_s"] = 8 * c.n_words / (ms / 1000.0)
        out[f"{name}_one_seed_per_letter_ms"] = one_ms
        out[f"{name}_cost_per_point_over_one_render"] = ms / (8 * one_ms)
    return out


def cull_config(kl, dev, flush):
    """Culled renders (kl_params.cull = 1): the same images with whole blocks
    of words placed at once where a closed-form disk bound certifies their
    pixel.  Gasket length 18 at 4096^2 (mixed and FP64) and the near-cusp
    group at length 20, 8192^2 (mixed).  Each culled image is compared bit for
    bit with the per-word render on the same prefix/suffix split, and timed
    against the per-word render on its default split.  Throughput is in
    word-equivalents/s: the words whose pixels the render fixes, not words
    evaluated one by one."""
    import torch

    def timed(r, K=7):
        for _ in range(2):
            r()
        ms = []
        for k in range(K):
            flush.fill_(k & 0xFF)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            r()
            b.record()
            torch.cuda.synchronize(dev)
            ms.append(a.elapsed_time(b))
        return statistics.median(ms)

    out = {}
    for tag, cfg, prec in (("gasket_d18_mixed", klsynth.C2, kl.MIXED),
                           ("gasket_d18_fp64", klsynth.C2, kl.FP64),
                           ("nearcusp_d20_mixed", klsynth.C3, kl.MIXED)):
        mk = lambda **f: kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width,
                                        cfg.height, cfg.window, prec, **f)
        rc = kl.Renderer(mk(cull=1), device=dev)
        cull_ms = timed(rc)
        sl = cfg.depth - 1 if cfg.depth - 1 <= 9 else min(12, max(9, cfg.depth // 2 + 1))
        rs = kl.Renderer(mk(prefix_len=cfg.depth - sl), device=dev)
        rs()
        same = bool(torch.equal(rc.image, rs.image) and
                    torch.equal(rc.counters[:3], rs.counters[:3]))
        del rs
        rw = kl.Renderer(mk(), device=dev)
        word_ms = timed(rw)
        del rw
        out[tag] = {"words": cfg.n_words, "culled_ms": cull_ms, "per_word_ms": word_ms,
                    "word_equivalents_per_s": cfg.n_words / (cull_ms / 1000.0),
                    "speedup_over_per_word": word_ms / cull_ms,
                    "identical_to_per_word_same_split": same,
                    "fp64_words": int(rc.counters[2].item())}
        del rc
    return out


def batch_sweep(kl, dev, steps: int):
    """The batched sweep: 256 seeded groups, depth 12..18, 1024^2 each, mixed,
    with launch shapes from the autotuner, captured once in a CUDA graph and
    replayed.  The images (1 GiB) exceed L2, so no flush is needed."""
    import torch
    from paper_1709_08018_gb300 import autotune
    cfgs = klsynth.batch_configs(256)
    ps = [kl.params_init(c.group.ta, c.group.tb, c.depth, c.width, c.height, c.window, kl.MIXED)
          for c in cfgs]
    t0 = time.time()
    tuned = autotune.tune_batch(ps, "sweep256-d12..18-1024", budget_s=45.0, repeats=2)
    tune_s = time.time() - t0
    b = kl.Batch(autotune.apply_batch(ps, tuned["best"]), device=dev)
    b.capture()
    for _ in range(2):
        b.replay()
    torch.cuda.synchronize(dev)
    K = max(3, min(steps, 10))
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(K)]
    for a, e in ev:
        a.record()
        b.replay()
        e.record()
    torch.cuda.synchronize(dev)
    ms = [a.elapsed_time(e) for a, e in ev]
    words = sum(c.n_words for c in cfgs)
    cnt = b.counters.cpu()
    assert int(cnt[:, 0].sum() + cnt[:, 1].sum()) == words
    out = {"workload": "256 groups, Re t in U[2,3], Im t in U[-0.05,0.05], depth U{12..18}, "
                       "1024^2 uint32 each over [-1.5,1.5]^2, mixed, one persistent launch "
                       "in a captured CUDA graph",
           "words_per_replay": words, "ms_per_replay": statistics.mean(ms),
           "words_per_s": words / (statistics.mean(ms) / 1000.0),
           "tuned": tuned["best"], "tune_seconds": tune_s, "candidates": len(tuned["tried"]),
           "fp64_words": int(cnt[:, 2].sum()), "replays": K}
    # the same sweep culled (kl_params.cull = 1): every word placed, each
    # group's image equal to its culled single render (tests/test_gpu_cull.py)
    pc = [kl.params_init(c.group.ta, c.group.tb, c.depth, c.width, c.height, c.window,
                         kl.MIXED, cull=1) for c in cfgs]
    bc = kl.Batch(pc, device=dev)
    bc.capture()
    for _ in range(2):
        bc.replay()
    torch.cuda.synchronize(dev)
    evc = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(K)]
    for a, e in evc:
        a.record()
        bc.replay()
        e.record()
    torch.cuda.synchronize(dev)
    msc = statistics.mean(a.elapsed_time(e) for a, e in evc)
    cntc = bc.counters.cpu()
    assert int(cntc[:, 0].sum() + cntc[:, 1].sum()) == words
    occ_w, occ_c = b.images != 0, bc.images != 0
    inter = (occ_w & occ_c).flatten(1).sum(1).double()
    union = (occ_w | occ_c).flatten(1).sum(1).double().clamp(min=1)
    out["culled"] = {"ms_per_replay": msc, "word_equivalents_per_s": words / (msc / 1000.0),
                     "speedup_over_per_word": statistics.mean(ms) / msc,
                     "iou_min_vs_per_word": float((inter / union).min()),
                     "fp64_words": int(cntc[:, 2].sum())}
    del b, bc
    torch.cuda.synchronize(dev)
    return out


def lod_config(kl, n_train: int = 64, n_test: int = 16, n_valid: int = 8):
    """Learned level-of-detail pruning: the network trained by the library's
    kernels on exact depth-22 renders of n_train groups (seed 1710), its
    pruning setting chosen on n_valid validation groups (seed 1712, target
    IoU 0.9995), evaluated on n_test held-out groups (seed 1711) at 8192^2
    against the exact render."""
    import torch
    from paper_1709_08018_gb300 import lod
    d, size, lo, hi, extent, under = 22, 8192, 8, 15, 1.0 / 32, 32.0
    W = (-2.0, 2.0, -2.0, 2.0)
    mk = lambda g: kl.params_init(g.ta, g.tb, d, size, size, W, kl.MIXED)
    tr = [mk(g) for g, _ in klsynth.draw_groups(klsynth.LOD_TRAIN_SEED, n_train)]
    va = [mk(g) for g, _ in klsynth.draw_groups(klsynth.LOD_VALID_SEED, n_valid)]
    te = [mk(g) for g, _ in klsynth.draw_groups(klsynth.LOD_HELDOUT_SEED, n_test)]
    t0 = time.time()
    x, t = lod.make_dataset(tr, lo, hi, per_level=60_000, seed=3, extent=extent)
    t1 = time.time()
    mlp, losses = lod.train(x, t, steps=10000, batch=16384, lr=2e-3, seed=5, under=under)
    torch.cuda.synchronize()
    t2 = time.time()
    tuned = lod.tune_prune(va, mlp, lo, hi, target=0.9995)
    margin, edge, hi_r = tuned["margin"], tuned["edge"], tuned["hi"]
    evals = [lod.evaluate(p, mlp, lo, hi_r, margin, edge, repeats=3) for p in te]
    s = lod.summarize(evals)
    # the exact culled render of the same groups (no network; every word placed)
    cul_ms, cul_iou, cul_diff = 0.0, 1.0, 0
    for p in te:
        q = kl.Params.from_buffer_copy(p)
        q.cull = 1
        rc, rw = kl.Renderer(q), kl.Renderer(p)
        rw()
        cul_ms += lod.time_ms(lambda: rc(), 3)
        a, b = rw.image != 0, rc.image != 0
        union = int((a | b).sum())
        cul_iou = min(cul_iou, int((a & b).sum()) / union if union else 1.0)
        cul_diff += int((rw.image != rc.image).sum())
        del rc, rw
    s["culled"] = {"ms": cul_ms, "speedup_over_exact": s["exact_ms"] / cul_ms,
                   "iou_min_vs_exact": cul_iou, "pixels_differing_from_exact": cul_diff,
                   "pruned_speedup_over_culled": cul_ms / s["pruned_ms"],
                   "network_beats_culled": s["pruned_ms"] < cul_ms,
                   "reading": "the exact culled render certifies sub-pixel subtrees "
                              "without the network's losses; the network prunes whole "
                              "subtrees before any of their words or disks are computed "
                              "and hands the rest to the same culling engine"}
    s.update({"workload": f"{n_test} held-out groups (seed 1711), depth 22 "
                          f"({kl.word_count(d)} words each), 8192^2 over [-2,2]^2; network "
                          f"trained on {n_train} groups (seed 1710); pruning setting chosen "
                          f"on {n_valid} validation groups (seed 1712)",
              "levels": [lo, hi], "render_levels": [lo, hi_r], "label_extent_px": extent,
              "under_weight": under, "margin": margin, "edge_px": edge,
              "valid_settings": [{"margin": m, "edge_px": e, "hi": h, "iou_min": round(i, 6),
                                  "ms": round(t, 3)} for m, e, h, i, t in tuned["tried"]],
              "train_samples": int(x.shape[0]), "train_steps": 10000,
              "loss_first_last": [losses[0], losses[-1]], "label_seconds": t1 - t0,
              "train_seconds": t2 - t1,
              "words_per_s_pruned": n_test * kl.word_count(d) / (s["pruned_ms"] / 1000.0),
              "words_per_s_exact": n_test * kl.word_count(d) / (s["exact_ms"] / 1000.0)})
    return s


def make_barrier(world: int):
    """A barrier over all ranks (a no-op for one process)."""
    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
    return barrier


def make_max_over_ranks(world: int, device):
    """x -> the maximum of x over all ranks (all_reduce MAX on `device`)."""
    def max_over_ranks(x: float) -> float:
        if world == 1:
            return x
        import torch
        import torch.distributed as dist
        t = torch.tensor([x], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        return float(t.item())
    return max_over_ranks


def make_image_sum(world: int):
    """(image, counters) -> both summed element-wise over the ranks into rank
    0's tensors (one reduce each).  The uint32 hit counts travel as int32:
    two's-complement addition wraps exactly as uint32 addition does."""
    def image_sum(image, counters):
        if world == 1:
            return
        import torch.distributed as dist
        dist.reduce(image, dst=0, op=dist.ReduceOp.SUM)
        dist.reduce(counters, dst=0, op=dist.ReduceOp.SUM)
    return image_sum


def shard_fields(world: int, rank: int) -> dict:
    """kl_params fields of rank `rank`'s shard of a job split over `world`
    processes (none for one process)."""
    return {"shard_index": rank, "shard_count": world} if world > 1 else {}


def job_rate(job_words: int, steps: int, local_ms: float, max_over_ranks):
    """Whole-job throughput: `steps` steps of a job of job_words words (all
    ranks together); the job's time is the slowest rank's.  Returns (words/s,
    job milliseconds)."""
    total_ms = max_over_ranks(local_ms)
    return job_words * steps / (total_ms / 1000.0), total_ms


def events(stream, n):
    import torch
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(n)]
    for e in ev:
        e.record(stream)   # create the underlying CUDA events
    return ev


def l2_atomic_peak(dev, n_adds: int = 1 << 26, image_words: int = 64 << 20, reps: int = 5):
    """Measured ceiling for the image adds: 32-bit atomic adds per second at
    uniformly random addresses of a 256 MiB image (torch's index_add_, one
    atomic add per index), the median of `reps` timed calls after 3 warm-ups.
    The render's adds come in runs and hit far fewer lines, so this is the
    pessimistic (scattered) ceiling the atomic fraction is quoted against."""
    import torch
    img = torch.zeros(image_words, dtype=torch.int32, device=dev)
    g = torch.Generator(device=dev)
    g.manual_seed(1709)
    idx = torch.randint(0, image_words, (n_adds,), device=dev, generator=g)
    ones = torch.ones(n_adds, dtype=torch.int32, device=dev)
    stream = torch.cuda.current_stream(dev)
    for _ in range(3):
        img.index_add_(0, idx, ones)
    ev = events(stream, 2 * reps)
    for k in range(reps):
        ev[2 * k].record(stream)
        img.index_add_(0, idx, ones)
        ev[2 * k + 1].record(stream)
    torch.cuda.synchronize(dev)
    ms = statistics.median(ev[2 * k].elapsed_time(ev[2 * k + 1]) for k in range(reps))
    assert int(img.sum(dtype=torch.int64)) == (3 + reps) * n_adds
    del img, idx, ones
    return n_adds / (ms / 1000.0)


def timed_render(kl, r, flush, stream, K, dev, image_sum=None):
    """K renders, each after an L2 flush, timed with CUDA events on `stream`
    (step = the kl_render call, plus the image sum when given) and with the
    library's events around its per-word kernel.  Returns (step ms list,
    kernel ms list)."""
    import torch
    st0, st1, kn0, kn1 = events(stream, K), events(stream, K), events(stream, K), events(stream, K)
    torch.cuda.synchronize(dev)
    for k in range(K):
        flush.fill_(k & 0xFF)                   # L2 flush, outside the timed events
        kl.set_profile_events(kn0[k], kn1[k])
        st0[k].record(stream)
        r()
        if image_sum is not None:
            image_sum(r.image, r.counters)
        st1[k].record(stream)
    kl.set_profile_events()
    torch.cuda.synchronize(dev)
    return ([st0[k].elapsed_time(st1[k]) for k in range(K)],
            [kn0[k].elapsed_time(kn1[k]) for k in range(K)])


def fp_peaks():
    pk = peaks()
    sm_max = float(pk.get("sm_max_mhz", 2070.0))
    return (SMS * FP32_LANES_PER_SM * sm_max * 1e6 / 1e12,
            SMS * FP64_LANES_PER_SM * sm_max * 1e6 / 1e12)


def roofline_filter(words, kern_ms, wl, exact_ops, traffic_key):
    """FP64 and double-float renders: every word takes the FP32 filter, about
    one in 10^4 the exact map of `exact_ops` operations (not counted)."""
    fp32_peak = fp_peaks()[0]
    ach = words * FILTER_OPS_PER_WORD / (kern_ms / 1000.0) / 1e12
    return {"bound": "alu", "kernel": "render_words_kernel", "achieved": ach, "peak": fp32_peak,
            "unit": "T FP32-op/s", "frac": ach / fp32_peak,
            "peak_kind": "derived: 152 SMs x 128 FP32 lanes x max SM clock",
            "filter_ops_per_word": FILTER_OPS_PER_WORD, "ops_per_word": exact_ops,
            "traffic": traffic_for(traffic_key, wl), "kernel_ms": kern_ms}


def roofline64(words, kern_ms, wl):
    return roofline_filter(words, kern_ms, wl, FP64_OPS_PER_WORD, "render_words_kernel<fp64>")


def plain_fp64(kl, cfg, dev, flush, K=3):
    """The plain FP64 path, measured: the FP64 render of the job's words over a
    window so small that the FP32 filter certifies nothing (its constants leave
    their range), so every word takes the FP64 map.  Median of K renders."""
    import torch
    p = kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width, cfg.height,
                       (-1e-100, 1e-100, -1e-100, 1e-100), kl.FP64)
    r = kl.Renderer(p, device=dev)
    r()
    step_ms, kern_ms = timed_render(kl, r, flush, torch.cuda.current_stream(dev), K, dev)
    cnt = r.counters.cpu()
    assert int(cnt[0]) + int(cnt[1]) == cfg.n_words
    del r
    ms, kms = statistics.median(step_ms), statistics.median(kern_ms)
    ops = cfg.n_words * FP64_OPS_PER_WORD / (kms / 1000.0) / 1e12
    return {"ms_per_step": ms, "words_per_s": cfg.n_words / (ms / 1000.0), "kernel_ms": kms,
            "fp64_pipe_frac": ops / fp_peaks()[1], "ops_per_word": FP64_OPS_PER_WORD}


def roofline32(words_fp32, kern_ms, wl):
    fp32_peak = fp_peaks()[0]
    ach = words_fp32 * FP32_OPS_PER_WORD / (kern_ms / 1000.0) / 1e12
    return {"bound": "alu", "kernel": "render_mixed_kernel", "achieved": ach, "peak": fp32_peak,
            "unit": "T FP32-op/s", "frac": ach / fp32_peak,
            "peak_kind": "derived: 152 SMs x 128 FP32 lanes x max SM clock",
            "ops_per_word": FP32_OPS_PER_WORD,
            "traffic": traffic_for("render_mixed_kernel", wl), "kernel_ms": kern_ms}


def roofline_df(words_df, kern_ms, wl):
    return roofline_filter(words_df, kern_ms, wl, DF64_OPS_PER_WORD, "render_words_kernel<df64>")


def secondary(kl, cfg, prec, flush, stream, dev, K):
    """One more whole-job render timed like the headline (N = 1): its rates,
    the roofline of its per-word kernel, its atomics and its image (host copy)
    for the accuracy figures."""
    import numpy as np
    p = kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width, cfg.height,
                       cfg.window, prec)
    r = kl.Renderer(p, device=dev)
    for _ in range(3):
        r()
    step_ms, kern_ms = timed_render(kl, r, flush, stream, K, dev)
    ms, kms = statistics.median(step_ms), statistics.median(kern_ms)
    cnt = [int(x) for x in r.counters.cpu().tolist()]
    assert cnt[0] + cnt[1] == cfg.n_words
    name = {kl.FP64: "FP64",
            kl.MIXED: "mixed (FP32 per-word map, FP64 prefixes and fallback words)",
            kl.DF64: "double-float (per-word map in hi+lo float pairs on the FP32 pipe, "
                     "FP64 prefixes and fallback words)"}[prec]
    roof = (roofline64(cfg.n_words, kms, cfg.name) if prec == kl.FP64 else
            roofline_df(cfg.n_words - cnt[2], kms, cfg.name) if prec == kl.DF64 else
            roofline32(cfg.n_words - cnt[2], kms, cfg.name))
    out = {"workload": describe(cfg, name),
           "words_per_step": cfg.n_words, "ms_per_step": ms,
           "words_per_s": cfg.n_words / (ms / 1000.0), "steps": K, "roofline": roof,
           "counters": {"in_window": cnt[0], "dropped": cnt[1], "fp64_words": cnt[2],
                        "atomics": cnt[3]},
           "atomics_per_s": cnt[3] / (kms / 1000.0)}
    img = r.image.cpu().numpy().view(np.uint32).copy()
    del r
    return out, img


def graph_replay_ms(kl, cfg, prec, flush, dev, K):
    """Median step time of the same whole-job render captured once in a CUDA
    graph and replayed (the parts, combine and per-word launches with one
    host launch), L2 flushed before each replay like the direct steps."""
    import torch
    p = kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width, cfg.height,
                       cfg.window, prec)
    r = kl.Renderer(p, device=dev)
    r.capture()
    stream = torch.cuda.current_stream(dev)
    for _ in range(3):
        r.replay()
    ev = events(stream, 2 * K)
    for k in range(K):
        flush.fill_(k & 0xFF)
        ev[2 * k].record(stream)
        r.replay()
        ev[2 * k + 1].record(stream)
    torch.cuda.synchronize(dev)
    cnt = r.counters.cpu()
    assert int(cnt[0]) + int(cnt[1]) == cfg.n_words
    del r
    return statistics.median(ev[2 * k].elapsed_time(ev[2 * k + 1]) for k in range(K))


def eval_sample(kl, cfg, prec, dev):
    """GPU pixel coordinates (kl_eval_words) of the seeded index sample."""
    import numpy as np
    import torch
    idx = klsynth.index_sample(klsynth.SAMPLE_SEED, SAMPLE_N, cfg.depth)
    p = kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width, cfg.height,
                       cfg.window, prec)
    t = torch.from_numpy(np.ascontiguousarray(idx).view(np.int64)).to(dev)
    return kl.eval_words(p, t).cpu().numpy()


def run_ours(args):
    import numpy as np
    import torch
    import paper_1709_08018_gb300 as kl

    world, rank, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    cfg, config = workload(world)
    N = cfg.n_words

    barrier = make_barrier(world)
    max_over_ranks = make_max_over_ranks(world, dev)
    image_sum = make_image_sum(world)

    p = kl.params_init(cfg.group.ta, cfg.group.tb, cfg.depth, cfg.width, cfg.height,
                       cfg.window, kl.FP64, **shard_fields(world, rank))
    r = kl.Renderer(p, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    stream = torch.cuda.current_stream(dev)

    for _ in range(args.warmup):
        r()
        image_sum(r.image, r.counters)
    torch.cuda.synchronize(dev)

    K = args.steps
    sampler = ClockSampler(local)
    with sampler:
        barrier()
        step_ms, kern_ms = timed_render(kl, r, flush, stream, K, dev, image_sum)
        barrier()
    clocks = sampler.summary()
    value, total_ms = job_rate(N, K, sum(step_ms), max_over_ranks)
    # one more render whose image and counters are summed: rank 0 holds the job's
    r()
    image_sum(r.image, r.counters)
    cnt = [int(x) for x in r.counters.cpu().tolist()]
    if rank == 0:
        assert cnt[0] + cnt[1] == N, cnt
    kern_s = statistics.mean(kern_ms) / 1000.0

    # end to end through the public API: host parameters in, the job's image
    # and counters copied back to pinned host memory every step (rank 0).  Two
    # image buffers: step k+1 renders while step k's image is copied out on a
    # second stream; the time is the span of all KE steps (CUDA events), L2
    # flushes included.
    rb = [r, kl.Renderer(p, device=dev)]
    host_img = [torch.empty((cfg.height, cfg.width), dtype=torch.int32, pin_memory=True)
                for _ in range(2)]
    host_cnt = [torch.empty(kl.KL_N_COUNTERS, dtype=torch.int64, pin_memory=True)
                for _ in range(2)]
    copy_stream = torch.cuda.Stream(dev)
    rendered = [torch.cuda.Event() for _ in range(2)]
    copied = [torch.cuda.Event() for _ in range(2)]
    KE = max(4, min(K, 10))
    e0, e1 = events(stream, 1)[0], events(stream, 1)[0]
    rb[1]()
    torch.cuda.synchronize(dev)
    barrier()
    e0.record(stream)
    for k in range(KE):
        b = k & 1
        flush.fill_(k & 0xFF)
        if k >= 2:
            stream.wait_event(copied[b])          # buffer b's previous image is out
        kl.render(rb[b].p, rb[b].image, rb[b].counters, rb[b].workspace, stream)
        image_sum(rb[b].image, rb[b].counters)
        rendered[b].record(stream)
        if rank == 0:
            copy_stream.wait_event(rendered[b])
            with torch.cuda.stream(copy_stream):
                host_img[b].copy_(rb[b].image, non_blocking=True)
                host_cnt[b].copy_(rb[b].counters, non_blocking=True)
        copied[b].record(copy_stream)
    stream.wait_event(copied[0])
    stream.wait_event(copied[1])
    e1.record(stream)
    torch.cuda.synchronize(dev)
    if rank == 0:
        for b in range(2):
            assert int(host_cnt[b][0]) + int(host_cnt[b][1]) == N
            hits = int(host_img[b].numpy().view(np.uint32).sum(dtype=np.uint64))
            assert hits == int(host_cnt[b][0]) % (1 << 64), (hits, int(host_cnt[b][0]))
    e2e_value, e2e_ms = job_rate(N, KE, e0.elapsed_time(e1), max_over_ranks)
    del rb, host_img

    line = {"metric": METRIC, "value": value, "unit": "words/s", "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": total_ms / K, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": config, "clocks": clocks,
            "roofline": dict(roofline64(N if world == 1 else N / world,
                                        statistics.mean(kern_ms), cfg.name),
                             kernel_share_of_step=statistics.mean(kern_ms) /
                             statistics.mean(step_ms)),
            "e2e": {"value": e2e_value, "unit": "words/s",
                    "h2d_bytes_per_step": __import__("ctypes").sizeof(r.p),
                    "d2h_bytes_per_step": cfg.width * cfg.height * 4 + kl.KL_N_COUNTERS * 8,
                    "overlap": "the copy of step k's image overlaps the render of step k+1 "
                               "(two image buffers, two streams)"},
            "gpu_launches": 3 * K,  # per step: parts, combine and the render kernel
            "counters": {"in_window": cnt[0], "dropped": cnt[1], "fp64_words": cnt[2],
                         "atomics": cnt[3]},
            "atomics_per_s": cnt[3] / world / kern_s}
    if world == 1:
        fp64_img = r.image.cpu().numpy().view(np.uint32).copy()
    del r
    torch.cuda.synchronize(dev)

    if world == 1:
        KS = max(5, min(K, 20))
        mixed3, mixed3_img = secondary(kl, klsynth.C3, kl.MIXED, flush, stream, dev, KS)
        # speedup_over_fp64: over the plain FP64 path (every word's map in FP64);
        # speedup_over_fp64_render: over the FP64 render, which filters in FP32 first
        line["plain_fp64"] = plain_fp64(kl, klsynth.C3, dev, flush)
        df3, df3_img = secondary(kl, klsynth.C3, kl.DF64, flush, stream, dev, KS)
        for v in (mixed3, df3):
            v["speedup_over_fp64"] = line["plain_fp64"]["ms_per_step"] / v["ms_per_step"]
            v["speedup_over_fp64_render"] = (total_ms / K) / v["ms_per_step"]
        mixed2, mixed2_img = secondary(kl, klsynth.C2, kl.MIXED, flush, stream, dev, KS)
        fp64_2, fp64_2_img = secondary(kl, klsynth.C2, kl.FP64, flush, stream, dev,
                                       max(3, KS // 4))
        plain2 = plain_fp64(kl, klsynth.C2, dev, flush)
        fp64_2["plain_fp64"] = plain2
        mixed2["speedup_over_fp64"] = plain2["ms_per_step"] / mixed2["ms_per_step"]
        mixed2["speedup_over_fp64_render"] = fp64_2["ms_per_step"] / mixed2["ms_per_step"]
        fp64_1, fp64_1_img = secondary(kl, klsynth.C1, kl.FP64, flush, stream, dev, KS)
        # the small job is launch-bound: the same render replayed from a graph
        gms = graph_replay_ms(kl, klsynth.C1, kl.FP64, flush, dev, KS)
        fp64_1["graph_replay"] = {"ms_per_step": gms,
                                  "words_per_s": klsynth.C1.n_words / (gms / 1000.0)}
        uv = {(c.name, prec): eval_sample(kl, c, prec, dev)
              for c in (klsynth.C3, klsynth.C2) for prec in (kl.FP64, kl.MIXED, kl.DF64)}
        if not args.no_cpu_baseline:
            # the oracle legs: the whole headline workload (the CPU baseline and
            # the reference image), the gasket render and the two samples
            ref3, secs3, threads = oracle_render(klsynth.C3)
            line["cpu_baseline"] = cpu_baseline(klsynth.C3, ref3, secs3, threads)
            t0 = time.perf_counter()
            idx3, z3 = oracle_sample(klsynth.C3)
            t1 = time.perf_counter() - t0
            # the paper-literal per-word definition on one core (d maps per word)
            line["cpu_baseline"]["per_word_one_thread"] = {
                "value": SAMPLE_N / t1, "unit": "words/s", "cores": 1,
                "sample": f"the seeded {SAMPLE_N}-index sample of the same workload, one orbit "
                          f"of {klsynth.C3.depth} maps per word, no binning"}
            line["accuracy"] = dict(image_agreement(fp64_img, ref3),
                                    **sample_dz(klsynth.C3, uv[(klsynth.C3.name, kl.FP64)], z3))
            mixed3["accuracy"] = dict(image_agreement(mixed3_img, ref3),
                                      **sample_dz(klsynth.C3, uv[(klsynth.C3.name, kl.MIXED)],
                                                  z3))
            df3["accuracy"] = dict(image_agreement(df3_img, ref3),
                                   **sample_dz(klsynth.C3, uv[(klsynth.C3.name, kl.DF64)], z3))
            del ref3
            ref2, _, _ = oracle_render(klsynth.C2)
            idx2, z2 = oracle_sample(klsynth.C2)
            mixed2["accuracy"] = dict(image_agreement(mixed2_img, ref2),
                                      **sample_dz(klsynth.C2, uv[(klsynth.C2.name, kl.MIXED)],
                                                  z2))
            fp64_2["accuracy"] = dict(image_agreement(fp64_2_img, ref2),
                                      **sample_dz(klsynth.C2, uv[(klsynth.C2.name, kl.FP64)],
                                                  z2))
            ref1, _, _ = oracle_render(klsynth.C1)
            fp64_1["accuracy"] = image_agreement(fp64_1_img, ref1)
            line["iou_vs_oracle"] = line["accuracy"]["iou_vs_oracle"]
            line["max_dz_rel"] = line["accuracy"]["max_dz_rel"]
            del ref2
        del fp64_img, mixed3_img, mixed2_img, fp64_2_img, fp64_1_img, df3_img
        line["df64_nearcusp_d20"] = df3
        line["mixed_nearcusp_d20"] = mixed3
        line["mixed_gasket_d18"] = mixed2
        # the image adds against a measured ceiling (scattered 32-bit atomic adds)
        peak = l2_atomic_peak(dev)
        line["l2_atomics"] = {
            "peak_per_s": peak,
            "peak_kind": "measured: torch index_add_ of 2^26 int32 adds at uniformly random "
                         "addresses of a 256 MiB buffer (one atomic add each)",
            "fp64_nearcusp_d20_frac": line["atomics_per_s"] / peak,
            "mixed_nearcusp_d20_frac": mixed3["atomics_per_s"] / peak,
            "mixed_gasket_d18_frac": mixed2["atomics_per_s"] / peak,
            "reading": "the ceiling is for scattered adds; the renders' adds come in runs "
                       "and bursts on nearby lines, and their kernels are bound by the FP32 "
                       "pipe and by issue, not by the L2"}
        line["fp64_gasket_d18"] = fp64_2
        line["fp64_gasket_d10"] = fp64_1
        if not args.no_tiling:
            line["tiling"] = tiling_config(kl, dev, K, flush)
        if not args.no_scan:
            line["paper_scan"] = scan_config(kl, dev, flush)
        if not args.no_maskit:
            line["maskit_example"] = maskit_config(kl, dev, flush)
        if not args.no_multiseed:
            line["multiseed"] = multiseed_config(kl, dev, flush)
        if not args.no_cull:
            line["culled"] = cull_config(kl, dev, flush)
        if not args.no_batch:
            line["batch_sweep"] = batch_sweep(kl, dev, K)
        if not args.no_lod:
            line["lod"] = lod_config(kl)
            line["lod"]["speedup_over_plain_fp64"] = (
                line["lod"]["words_per_s_pruned"] / plain2["words_per_s"])
            line["lod"]["speedup_over_fp64_render"] = (
                line["lod"]["words_per_s_pruned"] / fp64_2["words_per_s"])
    if rank == 0:
        print_line(line)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


# The headline and what it is checked with: on the line as they are.
EXACT_KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "config",
              "clocks", "roofline", "e2e", "cpu_baseline", "accuracy", "counters")
# Legs and tables of the stderr record alone.
SIDE_LEGS = ("fp64_gasket_d10", "paper_scan", "maskit_example", "multiseed")
TABLES = ("valid_settings", "per_group")


def short(x):
    """x with floats rounded to 6 significant digits, without its descriptions
    (texts of more than 45 letters) and tables."""
    if isinstance(x, float):
        return float(f"{x:.6g}")
    if isinstance(x, dict):
        return {k: short(v) for k, v in x.items()
                if k not in TABLES and not (isinstance(v, str) and len(v) > 45)}
    return [short(v) for v in x] if isinstance(x, (list, tuple)) else x


def print_line(line):
    """The result as one line on stdout, short enough for a reader that keeps 8,000
    letters; the whole record, descriptions and tables too, as one on stderr."""
    print(json.dumps(line), file=sys.stderr, flush=True)
    print(json.dumps({k: v if k in EXACT_KEYS else short(v) for k, v in line.items()
                      if k not in SIDE_LEGS}), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
