"""Autotuner for the query launch shapes.

Picks, for one index and one representative batch, the query path (separate
prefix/probe/expand launches, the persistent fused launch with
length-bucketed queues, region-binned probing, or content-ordered segments),
the segment length, the probe grid (CTAs per SM), the minimum k-mers a
warp takes, the fused path's tile size and short-query threshold, and the
expansion grid and byte-table policy.  It times the batch under each
candidate with CUDA events on the launching stream and insists that every
candidate returns exactly the same answer bits as the first one (the knobs
change launch shapes only).  Search: for every query path that this index
geometry and batch actually run (a requested path the library does not take
for them falls back to another, and is then not a separate candidate), a
coordinate descent over the other knobs, one knob at a time in the order of
KNOBS, keeping the best value before moving on, repeated while a whole pass
still improves (at most three passes); the best of the paths wins.
Knobs of a path that does not run (the fused path's tile and short-query
threshold, the binned path's regions) are not varied.
"""
from __future__ import annotations

import json
import os

# Tunings found on GB300, keyed by index geometry and batch shape.
CACHE_FILE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "tuning_cache.json")

KNOBS = (
    ("query_path", (0, 1, 2, 3)),
    ("branch_priority", (0, 1, 2)),
    ("use_byte_table", (0, 1)),
    ("expand_ctas_per_sm", (2, 4, 8, 16, 32)),
    # staged gathers before the fused grid: they pay off at a smaller grid
    # that leaves room for the k-mer branch beside it
    ("fused_async", (0, 1)),
    ("probe_ctas_per_sm", (0, 1, 2, 4, 8)),
    ("bin_region_kib", (16384, 32768, 65536, 131072)),
    ("bin_rows", (1, 2, 4)),
    ("seg_cut_bits", (4, 5, 6, 7, 8)),
    ("fused_tile_kmers", (256, 512, 1024, 2048, 4096)),
    ("fused_short_max", (64, 256, 1024, 4096)),
    ("probe_min_kmers_per_warp", (0, 256, 1024, 4096)),
)


def _time(run, reps: int):
    import torch
    stream = torch.cuda.current_stream()
    run()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(reps):
        e0.record(stream)
        run()
        e1.record(stream)
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best


def effective_path(tuning, info) -> int:
    """Sequence query path that this tuning and geometry ask for (the binding
    always passes a workspace large enough for paths 2 and 3, and batches as CSR
    offsets): the binned path for groups of at most 64 bytes, the content-ordered
    path for groups of at most 64 bytes and eta <= 4, the fused path for groups of
    at most 512 bytes, else the separate launches.  The library runs the fused
    path's small batches and one-lane groups as separate launches too, by rules on
    the batch: `ran_path` tells from the launches."""
    g = info["group_bytes"]
    if tuning["query_path"] == 2 and g <= 64:
        return 2
    if tuning["query_path"] == 3 and g <= 64 and info.get("eta", 1) <= 4:
        return 3
    if tuning["query_path"] >= 1 and g <= 512:
        return 1
    return 0


def ran_path(path: int, profile) -> int:
    """`path` (of effective_path) as the library ran it, from the launch counts
    since a profile_reset: the persistent launch expands its own answers, the
    separate launches have an expansion.  (Groups that reach the fused path
    answer single k-mers without one.)"""
    return 0 if path == 1 and profile["expand"]["launches"] else path


def _path_of(idx, run, start) -> int:
    """The path that the batch takes under the tuning `start`."""
    path = effective_path(start, idx.info)
    if path != 1 or not hasattr(idx, "profile_reset"):
        return path
    idx.set_tuning(**start)
    idx.profile_reset()
    run()
    idx.sync()
    return ran_path(path, idx.profile_read())


def _descend(idx, run, outputs, ref, start, path, knobs, reps, trials, verbose, passes: int = 3):
    """Coordinate descent from `start` over `knobs`, repeated while a whole
    pass still improves (at most `passes`: a knob tuned early may want
    another value once a later one has moved); returns (best, ms)."""
    import torch
    idx.set_tuning(**start)
    best_cfg, best_ms = dict(start), _time(run, reps)
    trials.append({"tuning": dict(start), "ms": best_ms})
    for _ in range(passes):
        before = dict(best_cfg)
        best_cfg, best_ms = _one_pass(idx, run, outputs, ref, best_cfg, best_ms, knobs, reps, path, trials,
                                      verbose)
        if best_cfg == before:
            break
    return best_cfg, best_ms


def _one_pass(idx, run, outputs, ref, best_cfg, best_ms, knobs, reps, path, trials, verbose):
    import torch
    for knob, values in knobs:
        if knob in ("fused_tile_kmers", "fused_short_max", "fused_async") and path != 1:
            continue
        if knob in ("bin_region_kib", "bin_rows") and path != 2:
            continue
        if knob == "seg_cut_bits" and path != 3:
            continue
        for v in values:
            if best_cfg.get(knob) == v:
                continue
            cand = dict(best_cfg)
            cand[knob] = v
            idx.set_tuning(**cand)
            ms = _time(run, reps)
            idx.sync()
            for a, b in zip(ref, outputs()):
                if not torch.equal(a, b):
                    raise RuntimeError(f"tuning {cand} changed the answers")
            trials.append({"tuning": cand, "ms": ms})
            if verbose:
                print(f"autotune path {path} {knob}={v}: {ms:.4f} ms (best {best_ms:.4f})", flush=True)
            if ms < best_ms:
                best_cfg, best_ms = cand, ms
    return best_cfg, best_ms


def autotune(idx, run, outputs, reps: int = 7, knobs=KNOBS, verbose: bool = False) -> dict:
    """Tunes `idx` for the batch that `run()` enqueues on the current stream.

    `outputs()` returns the tensors holding the batch's answers after a run;
    every candidate's answers must equal the first run's bit for bit.
    Leaves the best tuning set on `idx` and returns
    {"best": tuning, "ms": best time, "trials": [...]}.
    """
    base = idx.get_tuning()
    run()
    idx.sync()
    ref = [t.clone() for t in outputs()]
    paths = dict(knobs).get("query_path", (base["query_path"],))
    rest = [(k, v) for k, v in knobs if k != "query_path"]
    starts, seen = [], set()
    for qp in paths:
        start = dict(base, query_path=qp)
        path = _path_of(idx, run, start)
        if path not in seen:
            seen.add(path)
            starts.append((start, path))
    trials, best = [], None
    try:
        for start, path in starts:
            cfg, ms = _descend(idx, run, outputs, ref, start, path, rest, reps, trials, verbose)
            if best is None or ms < best[1]:
                best = (cfg, ms)
    except Exception:
        idx.set_tuning(**base)
        raise
    idx.set_tuning(**best[0])
    return {"best": best[0], "ms": best[1], "trials": trials}


def cache_key(idx, n_queries: int, n_kmers: int) -> str:
    i = idx.info
    return (f"K{i['K']}_B{i['B']}_R{i['R']}_m{i['m']}_eta{i['eta']}_k{i['k']}"
            f"_n{n_queries}_kpq{n_kmers // max(n_queries, 1)}")


def load_cached(path: str, key: str):
    try:
        with open(path) as f:
            return json.load(f).get(key)
    except Exception:
        return None


def store_cached(path: str, key: str, tuning: dict):
    data = {}
    try:
        with open(path) as f:
            data = json.load(f)
    except Exception:
        pass
    data[key] = tuning
    os.makedirs(os.path.dirname(os.path.abspath(path)), exist_ok=True)
    with open(path, "w") as f:
        json.dump(data, f, indent=1, sort_keys=True)
