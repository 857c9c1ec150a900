"""Branching in large instances under clause learning, where shared memory holds
a bound per 128 variables instead of the activities: the checked build compares
every decision with the full scan over the activities (and every index with its
buffer) and reports a difference as a failed check. Sizes: the activities in
shared memory, bounds beside the trail positions, bounds only; whole groups of
128 variables and a remainder of one. Each instance is a random 3-SAT core at
the threshold, whose variables lie anywhere among the others, and loose clauses
over the rest that any assignment search satisfies: its verdict is the core's."""
import json
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import json, sys
import numpy as np
sys.path.insert(0, ROOT)
sys.path.insert(0, ROOT + "/tests")
from paper_2601_21552_gb300 import api, binding as B
assert B.LIB_PATH.endswith("libscuba_checked.so"), B.LIB_PATH
from workloads import queries
from raw_cnf import model_ok, solve_raw
CORE = 130
out = []
for V in (2688, 2945, 4865, 6529):
    cores, large = [], []
    for seed in range(6):
        rng = np.random.default_rng([V, seed])
        n, l = queries.random_3sat(3100 + seed, CORE, CORE)
        core = [list(map(int, c)) for c in l]
        ids = rng.permutation(V) + 1
        place = lambda c: [int(np.sign(x)) * int(ids[abs(x) - 1]) for x in c]
        rest = ids[CORE:]
        # the rest all true satisfies every loose clause
        loose = [[int(a), -int(b), int(c)] for a, b, c in
                 (rng.choice(rest, 3, replace=False) for _ in range(2 * V))]
        cores.append((CORE, core))
        large.append((V, [place(c) for c in core] + loose))
    _, vc, _, _, _ = solve_raw(api, cores, search="dpll", time_budget_ms=30000)
    st, v, m, vb, _ = solve_raw(api, large, search="cdcl", time_budget_ms=30000)
    out.append({"V": V, "status": int(st), "msg": B.last_error(),
                "core": [int(x) for x in vc], "large": [int(x) for x in v],
                "models": bool(all(model_ok(large[i][1], m, vb[i])
                                   for i in range(len(large)) if v[i] == 1))})
print("RESULT " + json.dumps(out))
'''


def test_bounded_pick_equals_full_scan():
    from paper_2601_21552_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CHILD], timeout=300,
                       capture_output=True, text=True, cwd=ROOT,
                       env=dict(os.environ, SCUBA_LIBRARY="checked"))
    line = [x for x in r.stdout.splitlines() if x.startswith("RESULT ")]
    assert r.returncode == 0 and line, r.stdout[-2000:] + r.stderr[-2000:]
    for got in json.loads(line[0][7:]):
        assert got["status"] == 0, got
        assert got["large"] == got["core"] and set(got["core"]) <= {0, 1}, got
        assert got["models"], got
