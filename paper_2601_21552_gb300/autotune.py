"""Offline autotuner for the persistent search: launch shape and subtree
sharing parameters.

Sweeps blocks per SM, the decisions a subtree makes before it may share work
(split_min) and the decisions between checks for idle warps (split_interval)
on a workload, timing each setting over several solves, and writes the
setting with the lowest MEAN time. The workload is a large batch, on which
every warp starts busy, and two small ones, on which a few hard instances have
to reach the idle warps; settings are ranked by the geometric mean of the
batches' mean times (a steady setting within 5 % of the lowest wins over one
whose slowest solve of any batch took more than 1.5x that batch's median; tails
are judged and averaged batch by batch, since a mean over them would hide them) and written to a JSON file that bench.py and
api.solve(..., tuned=True) read. The search is nondeterministic: a few runs
in ten can take several times the median (a hard instance's cube tree grows
much deeper in them), so the mean -- what a sequence of solves costs -- is
the objective, over enough repetitions to see those runs.

    python -m paper_2601_21552_gb300.autotune [--queries 4096] [--width 16]
           [--reps N] [--search dpll|cdcl]
           [--out paper_2601_21552_gb300/autotune.json]

The DPLL sweep writes "best"; the clause-learning sweep (cube-sharing
thresholds and depth) writes "best_cdcl".
"""
from __future__ import annotations

import argparse
import itertools
import json
import os
import statistics
import sys
import time

HERE = os.path.dirname(os.path.abspath(__file__))
DEFAULT_OUT = os.path.join(HERE, "autotune.json")
SPACE = {
    "blocks_per_sm": [2, 3],
    "split_min": [64, 128],
    "split_interval": [16],
}
# clause learning: decisions before a job may give away cubes, the decisions
# between checks for idle warps (both while most warps are idle, see
# scuba_options) and the deepest cube level that may split further (248: the
# prefix capacity, no cap); split_min of 8 and less lets cube trees explode (10
# was measured within 1 % of 12), 24 and more leaves small batches waiting; the
# conflicts per Luby restart unit (25) come from a sweep over {12, 25, 40, 50,
# 100}; share_lbd is the LBD bound of the clauses the jobs of one instance share
# (-1: no sharing; reading fewer of them pays more than they prune, and deep cubes
# share two-level clauses in any case); a gate
# on the job's own conflicts before it may give cubes away (8-128) was measured no better
# than none
SPACE_CDCL = {
    "split_min": [12, 16],
    "split_depth": [248],
    "split_interval": [4, 8],
    "restart_unit": [25],
    "share_lbd": [1, 2],
}


def load(path: str = DEFAULT_OUT, section: str = "best") -> dict:
    """Best options found by a previous sweep ("best": the DPLL search,
    "best_cdcl": the clause-learning search), or {} when none was run."""
    try:
        with open(path) as f:
            return dict(json.load(f).get(section, {}))
    except (OSError, ValueError):
        return {}


def sweep(db, reps: int = 3, space: dict | None = None, time_budget_ms: int = 120000,
          fixed: dict | None = None, more: tuple = ()):
    """Times every setting of `space` on db and each batch of `more`, reps solves
    each; a setting's mean and median are the geometric means of its batches'.
    Returns (the choice, all trials)."""
    import numpy as np
    import torch

    from . import api
    space = space or SPACE
    keys = list(space)
    trials = []
    for combo in itertools.product(*(space[k] for k in keys)):
        opts = dict(zip(keys, combo))
        batches = (db, *more)
        times, failed = [[] for _ in batches], []
        for _ in range(reps):
            for batch, each in zip(batches, times):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                api.solve(batch, want_model=False, stats=False, time_budget_ms=time_budget_ms,
                          **opts, **(fixed or {}))
                rc = api.status()
                each.append(time.perf_counter() - t0 if rc == 0 else float("inf"))
                if rc != 0:
                    failed.append(rc)  # e.g. the time budget reached
        over = lambda stat: float(np.exp(np.mean(np.log([stat(t) for t in times]))))
        trials.append({"options": opts, "mean_s": over(np.mean), "median_s": over(np.median),
                       "times": times if more else times[0]})
        if failed:
            trials[-1]["failed_status"] = failed
        print(json.dumps(trials[-1]), flush=True)
    return pick(trials), trials


def pick(trials, within: float = 0.05, tail: float = 1.5):
    """The trial with the lowest mean time, unless its slowest solve took more
    than `tail` times the median of its batch (a setting prone to the rare
    several-times-slower solve) and a steady trial lies within `within` of that
    mean: then the steady trial with the lowest mean. A trial's times are one
    batch's, or a list of each batch's."""
    def is_steady(times):
        batches = times if isinstance(times[0], (list, tuple)) else [times]
        return all(max(t) <= tail * statistics.median(t) for t in batches)

    best = min(trials, key=lambda t: t["mean_s"])
    steady = [t for t in trials if t["mean_s"] <= best["mean_s"] * (1.0 + within)
              and is_steady(t["times"])]
    return min(steady, key=lambda t: t["mean_s"]) if steady else best


def summary(trial):
    """A trial as the file keeps it: of each batch's solves the mean, the median
    and the slowest (every tuned call reads the file, so it stays small)."""
    batches = [{"mean_s": round(statistics.fmean(t), 6), "median_s": round(statistics.median(t), 6),
                "max_s": round(max(t), 6)} for t in trial["times"]]
    rest = {k: v for k, v in trial.items() if k != "times"}
    return {**rest, "mean_s": round(trial["mean_s"], 6),
            "median_s": round(trial["median_s"], 6), "batches": batches}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--queries", type=int, default=4096)
    ap.add_argument("--width", type=int, default=16)
    ap.add_argument("--reps", type=int, default=0, help="solves per setting (0: 16)")
    ap.add_argument("--out", default=DEFAULT_OUT)
    ap.add_argument("--search", default="dpll", choices=["dpll", "cdcl"])
    ap.add_argument("--space", default="", help="JSON dict replacing the sweep space, "
                    "e.g. '{\"split_min\": [8, 16], \"split_depth\": [12, 14]}'")
    args = ap.parse_args()
    args.reps = args.reps or 16
    sys.path.insert(0, os.path.dirname(HERE))
    import torch

    from . import api, binding as B
    from workloads import queries
    irs, _ = queries.config2(args.queries, w=args.width)
    enc = B.scuba_encode_batch(irs)
    db = api.DeviceBatch(enc, "cuda")
    more = tuple(api.DeviceBatch(B.scuba_encode_batch(q), "cuda") for q in
                 (queries.config1(256, w=8)[0], queries.config2(512, w=10)[0]))
    torch.cuda.synchronize()
    space = json.loads(args.space) if args.space else None
    if args.search == "cdcl":
        best, trials = sweep(db, reps=args.reps, space=space or SPACE_CDCL,
                             fixed={"search": "cdcl"}, more=more)
    else:
        best, trials = sweep(db, reps=args.reps, space=space, more=more)
    try:  # the other search's section stays as it was
        with open(args.out) as f:
            out = json.load(f)
    except (OSError, ValueError):
        out = {}
    sfx = "_cdcl" if args.search == "cdcl" else ""
    out.update({"workload": f"partition queries, {args.width}-bit inputs, {args.queries} queries; "
                            "256 bounds queries of 8 bits; 512 partition queries of 10 bits",
                "device": torch.cuda.get_device_name(0), "reps" + sfx: args.reps,
                "best" + sfx: best["options"], "best_mean_s" + sfx: best["mean_s"],
                "best_median_s" + sfx: best["median_s"],
                "trials" + sfx: [summary(t) for t in trials]})
    with open(args.out, "w") as f:
        json.dump(out, f)
    print("best", json.dumps(best))


if __name__ == "__main__":
    main()
