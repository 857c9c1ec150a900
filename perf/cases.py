"""The work a user of this framework has it do, case by case.

A case names one call through the public entry points (``api``, ``binding``,
``frontend``) together with its sizes; ``prepare`` builds what a program holds
before that call and ``run`` makes the call. The families are the ones of the
bench and the tests: bounds and partition queries of 8 to 16 bits, queries
grown with 2-D/3-D ids and cubic sizes, random 3-SAT, stencil kernels in the
incremental form, unit-propagation closures, and the branching network.

Satisfying assignments are not returned: every call asks for them (that work
is part of the pass), but any assignment that satisfies the formula is a right
answer and the search's order of parallel work decides which one is found.
Verdicts, closures and gradients are returned whole.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2601_21552_gb300 import api, binding as B, frontend
from paper_2601_21552_gb300.frontend import IR

TIME_MS = 60000  # time budget of a solve: far above what any case takes

# network sizes and parameter layout, as include/scuba.h states them
FEATURES, HIDDEN = 16, 64
MOST_ROWS = 2000  # rows of a decision node: its open variables


def listed():
    return [
        # the accesses of one small kernel checked on their own: latency counts
        {"name": "check_bounds8_12", "kind": "cdcl", "family": "bounds", "width": 8, "count": 12},
        # a whole program's 1-D bounds queries, the bench's first configuration
        {"name": "check_bounds8_256", "kind": "cdcl", "family": "bounds", "width": 8, "count": 256},
        # the bench's default workload: a large batch of partition queries
        {"name": "check_partition16_4096", "kind": "cdcl", "family": "partition", "width": 16,
         "count": 4096},
        # DIMACS-style input that the encoder did not write: random 3-SAT at the threshold
        {"name": "check_3sat150_511", "kind": "cdcl", "family": "3sat", "width": 150, "count": 511},
        # large uneven queries: 2-D/3-D ids and cubic sizes, no path condition
        {"name": "check_grown_128", "kind": "cdcl", "family": "grown", "width": 0, "count": 128},
        # the library's default search (no clause learning) on a program's queries
        {"name": "dpll_bounds8_256", "kind": "dpll", "family": "bounds", "width": 8, "count": 256},
        # learned branching: the network scores the top decisions of the search
        {"name": "learned_partition10_512", "kind": "learned", "family": "partition", "width": 10,
         "count": 512},
        # one shared query per kernel, its accesses as units under selector assumptions
        {"name": "units_stencil8_48", "kind": "units", "family": "stencil", "width": 8, "count": 48},
        # what a launch's constants settle by unit propagation alone, no search
        {"name": "close_partition16_4096", "kind": "close", "family": "partition", "width": 16,
         "count": 4096},
        # the same for a few large uneven queries
        {"name": "close_grown_33", "kind": "close", "family": "grown", "width": 0, "count": 33},
        # loss and gradient of one training minibatch: 64 decision nodes
        {"name": "gradient_64", "kind": "gradient", "family": "trace", "width": 0, "count": 64},
        # the same over a whole recorded trace (held-out loss, full-batch steps)
        {"name": "gradient_1001", "kind": "gradient", "family": "trace", "width": 0,
         "count": 1001},
    ]


def draw(rng):
    def spread(lo, hi):  # log-uniform whole number, odd ones among them
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["cdcl", "cdcl", "cdcl", "cdcl", "dpll", "learned", "units", "close",
                       "close", "gradient", "gradient"])
    if kind == "cdcl":
        family = rng.choice(["bounds", "partition", "3sat", "grown"])
        if family == "3sat":
            return {"kind": kind, "family": family, "width": rng.randint(50, 150),
                    "count": spread(24, 511)}
        if family == "grown":
            return {"kind": kind, "family": family, "width": 0, "count": spread(24, 128)}
        return {"kind": kind, "family": family, "width": rng.randint(6, 14),
                "count": spread(12 if family == "bounds" else 48, 4096)}
    if kind in ("dpll", "learned"):
        family = rng.choice(["bounds", "partition"])
        return {"kind": kind, "family": family,
                "width": rng.randint(6, 10 if kind == "dpll" else 9),
                "count": spread(12 if family == "bounds" else 48, 512)}
    if kind == "units":
        return {"kind": kind, "family": "stencil", "width": rng.randint(6, 8),
                "count": spread(4, 48)}
    if kind == "close":
        family = rng.choice(["bounds", "partition", "grown"])
        if family == "grown":
            return {"kind": kind, "family": family, "width": 0, "count": spread(4, 256)}
        return {"kind": kind, "family": family, "width": rng.randint(6, 16),
                "count": spread(12, 4096)}
    return {"kind": kind, "family": "trace", "width": 0, "count": spread(8, 1001)}


# ---------------------------------------------------------------------------
# Queries
# ---------------------------------------------------------------------------

def bounds_ir(r, w):
    """offset = a*(bid*bdim + tid) + c against size = k1*n + k0, guarded by
    idx < n in half of the queries."""
    ir = IR()
    n, tid, bid, bdim = (ir.free(w, x) for x in ("n", "tid", "bid", "bdim"))
    idx = ir.add(ir.mul(bid, bdim), tid)
    offset = ir.add(ir.mul(ir.const(r.integers(1, 5)), idx), ir.const(r.integers(0, 8)))
    size = ir.add(ir.mul(ir.const(r.integers(1, 5)), n), ir.const(r.integers(0, 8)))
    ir.assert_(ir.ult(tid, bdim))
    if r.random() < 0.5:
        ir.assert_(ir.ult(idx, n))
    ir.assert_(ir.ule(size, offset))
    return ir.to_array()


def partition_ir(r, w):
    """One allocation of k1*n + k0 elements split at i*(n/k); the access goes
    to partition j."""
    ir = IR()
    n, tid, bid, bdim = (ir.free(w, x) for x in ("n", "tid", "bid", "bdim"))
    idx = ir.add(ir.mul(bid, bdim), tid)
    size = ir.add(ir.mul(ir.const(r.integers(1, 5)), n), ir.const(r.integers(0, 8)))
    k = int(r.integers(2, 9))
    j = int(r.integers(0, k))
    m = ir.udiv(n, k)
    p_j = ir.mul(ir.const(j), m)
    end_j = ir.mul(ir.const(j + 1), m) if j < k - 1 else size
    offset = ir.add(p_j, ir.add(ir.mul(ir.const(r.integers(1, 5)), idx),
                                ir.const(r.integers(0, 8))))
    ir.assert_(ir.ult(tid, bdim))
    if r.random() < 0.5:
        ir.assert_(ir.ult(idx, m))
    ir.assert_(ir.or_(ir.ult(offset, p_j), ir.ule(end_j, offset)))
    return ir.to_array()


def grown_ir(r):
    """A bounds query of 8, 16 or 32 bits grown by further id dimensions,
    row-major scalings and cubic size factors up to a log-uniform size; one
    query in three stays a plain 8-bit bounds query, guarded or not."""
    if r.random() < 0.33:
        return bounds_ir(r, 8)
    w = int(r.choice([8, 16, 32], p=[0.4, 0.4, 0.2]))
    cells = math.exp(r.uniform(math.log(500), math.log(200000))) / 14  # bit cells to spend
    ir = IR()
    n, tid, bid, bdim = (ir.free(w, x) for x in ("n", "tid", "bid", "bdim"))
    ir.assert_(ir.ult(tid, bdim))
    idx = ir.add(ir.mul(bid, bdim), tid)
    size = ir.add(ir.mul(ir.const(r.integers(1, 5)), n), ir.const(r.integers(0, 8)))
    w_idx, w_size = 2 * w + 1, w + 3
    cells -= w * w + 6 * w
    while True:
        what = int(r.integers(0, 3))
        if what == 2:  # (N + 1)^3 * E * 3
            wf = 4 * w + 5
            cost = 3 * (w + 1) ** 2 + (3 * w + 3) * w + 2 * wf + w_size * wf
        else:          # idx * x + t, size * x
            cost = (w_idx + w_size) * w + 4 * w
        if cost > cells:
            break
        cells -= cost
        if what == 2:
            big_n, e = ir.free(w, "N"), ir.free(w, "E")
            n1 = ir.add(big_n, ir.const(1))
            f = ir.mul(ir.mul(ir.mul(ir.mul(n1, n1), n1), e), ir.const(3))
            size = ir.mul(size, f)
            w_size += wf
        else:
            bd, t = ir.free(w, "bd"), ir.free(w, "t")
            ir.assert_(ir.ult(t, bd))
            idx = ir.add(ir.mul(idx, bd), t)
            size = ir.mul(size, bd)
            w_idx, w_size = w_idx + w + 1, w_size + w
    offset = ir.add(ir.mul(ir.const(r.integers(1, 5)), idx), ir.const(r.integers(0, 8)))
    ir.assert_(ir.ule(size, offset))
    return ir.to_array()


def stencil_text(r, w):
    """A 1-D stencil kernel: neighbours under a guard that may be too weak for
    the farthest of them, some without a guard."""
    radius, block = 3, 1 << int(r.integers(4, 7))
    inside = "\n".join("    access a[idx %s %d]" % ("+" if d >= 0 else "-", abs(d))
                       for d in range(-radius, radius + 1))
    slack, reach = int(r.integers(0, 3)), int(r.integers(0, 5))
    return f"""input n {w}
input bd {w}
malloc buf n + {slack}
launch stencil grid((n + {block - 1}) / {block}) block(bd) args(buf, n)
kernel stencil(a, m)
  let idx = blockIdx.x * blockDim.x + threadIdx.x
  if idx >= {reach} && idx + {reach} < m
{inside}
  end
  access a[idx + {radius}]
  if idx < m
    access a[idx]
    access a[m - idx - {reach}]
  end
end
"""


def random_3sat(r, nv):
    """Uniform random 3-SAT at 4.26 clauses per variable: int32 [m, 3]."""
    m = int(round(4.26 * nv))
    a = r.integers(0, nv, m)
    b = (a + r.integers(1, nv, m)) % nv
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    c = r.integers(0, nv - 2, m)  # skip the two variables already taken
    c = c + (c >= lo)
    c = c + (c >= hi)
    v = np.stack([a, b, c], axis=1) + 1
    return np.where(r.random((m, 3)) < 0.5, v, -v).astype(np.int32)


def irs_of(case, r):
    make = {"bounds": lambda: bounds_ir(r, case["width"]),
            "partition": lambda: partition_ir(r, case["width"]),
            "grown": lambda: grown_ir(r)}[case["family"]]
    return [make() for _ in range(case["count"])]


def sat_batch(case, r):
    cnfs = [random_3sat(r, case["width"]) for _ in range(case["count"])]
    per = np.array([len(c) for c in cnfs], np.int64)
    icb = np.concatenate([[0], np.cumsum(per)]).astype(np.int64)
    nv = np.full(case["count"], case["width"], np.int32)
    vb = np.concatenate([[0], np.cumsum(nv)]).astype(np.int64)
    return api.DeviceBatch.from_csr(icb, 3 * np.arange(icb[-1] + 1, dtype=np.int64),
                                    np.concatenate(cnfs).reshape(-1), nv, vb)


def launch_constants(enc, r, w_of):
    """Assumption literals that fix the size input, the thread id and the
    block dimension (a power of two above the thread id) of every query and
    leave the block id open: (asm_begin, asm_lits)."""
    iib, widths, var = enc.inputs()
    bit0 = np.concatenate([[0], np.cumsum(widths)]).astype(np.int64)
    begin, lits = [0], []
    for i in range(enc.n):
        w = w_of(widths[iib[i]])
        bdim = 1 << int(r.integers(1, w - 1))
        fixed = {0: int(r.integers(1 << (w - 1), 1 << w)), 1: int(r.integers(0, bdim)), 3: bdim}
        for word, value in fixed.items():
            at = bit0[iib[i] + word]
            lits += [int(var[at + k]) if value >> k & 1 else -int(var[at + k])
                     for k in range(int(widths[iib[i] + word]))]
        begin.append(len(lits))
    return np.array(begin, np.int64), np.array(lits, np.int32)


def most_vars(case):
    """Room for the closures of any batch of this case: about 100 variables
    per bit of a bounds or partition query, 50,000 of the largest grown one."""
    return case["count"] * (50000 if case["family"] == "grown" else 160 * case["width"])


# ---------------------------------------------------------------------------
# Decision traces
# ---------------------------------------------------------------------------

def features(rows, depth, assigned, g):
    """Rows of the 16 features of the residual formula in the ranges the
    search records them (BF16 on the device)."""
    dev = "cuda"
    u = torch.rand((rows, 8), generator=g, device=dev)
    c2p, c3p, c2n, c3n = (torch.floor(-torch.log1p(-u[:, k] * 0.999) * s)
                          for k, s in enumerate((1.0, 2.5, 1.0, 2.5)))
    op, on = c2p + c3p + torch.floor(3 * u[:, 4]), c2n + c3n + torch.floor(3 * u[:, 5])
    act = torch.clamp(-torch.log1p(-u[:, 6] * 0.999) * 0.1 - 0.1, 0, 1)
    inp = (u[:, 7] < 0.04).float()
    x = torch.stack([c2p / 4, c3p / 4, c2n / 4, c3n / 4, op / 8, on / 8, act, inp,
                     inp * u[:, 7] * 25, depth, assigned, (c2p + c2n) / 8, (c3p + c3n) / 8,
                     torch.log2(1 + op + on) / 6, (c2p + c3p - c2n - c3n) / 8,
                     torch.ones_like(act)], dim=1)
    return x.to(torch.bfloat16)


def node_rows(case, r):
    """Rows of each decision node: what is still open of 300 to
    MOST_ROWS variables."""
    return np.exp(r.uniform(math.log(300), math.log(MOST_ROWS), case["count"])).astype(np.int64)


def make_trace(case, seed):
    r = np.random.default_rng([seed, 9])
    g = torch.Generator(device="cuda").manual_seed(seed)
    nrows = node_rows(case, r)
    rows = int(nrows.sum())
    n = torch.from_numpy(nrows).cuda()
    per = lambda v: torch.repeat_interleave(torch.from_numpy(v).float().cuda(), n, output_size=rows)
    x = features(rows, per(r.integers(0, 8, len(nrows)) / 32.0), per(r.random(len(nrows)) * 0.5), g)
    u = torch.rand(rows, generator=g, device="cuda")
    target = torch.where(u < 0.7, 0.0, torch.floor(1 - 8 * torch.log((1 - u) / 0.3 + 1e-3)))
    closed = torch.from_numpy((r.random(len(nrows)) < 0.98).astype(np.int32)).cuda()
    tr = api.Trace(8, len(nrows), MOST_ROWS * len(nrows))  # a recorded trace leaves room too
    tr.x[:rows * FEATURES].copy_(x.view(torch.int16).reshape(-1))
    tr.target[:rows].copy_(target)
    tr.node_row.copy_(torch.cumsum(n, 0) - n)
    tr.node_nrows.copy_(n)
    tr.node_closed.copy_(closed)
    tr.counts.copy_(torch.tensor([len(nrows), rows]))
    return tr


# ---------------------------------------------------------------------------
# The interface
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    r = np.random.default_rng([seed, 3])
    if kind in ("cdcl", "dpll", "learned"):
        if case["family"] == "3sat":
            db = sat_batch(case, r)
        else:
            db = api.DeviceBatch(B.scuba_encode_batch(irs_of(case, r)))
        s = {"kind": kind, "db": db}
        if kind == "learned":  # a fixed network: how it was trained does not matter to a pass
            s["net"] = api.Mlp(seed=3)
        return s
    if kind == "units":
        kqs = [frontend.kernel_queries(frontend.parse(stencil_text(r, case["width"])),
                                       bid_width=case["width"])[0] for _ in range(case["count"])]
        enc = B.scuba_encode_batch([kq.ir for kq in kqs])
        iib, widths, var = enc.inputs()
        bit0 = np.concatenate([[0], np.cumsum(widths)]).astype(np.int64)
        unit_inst = [i for i, kq in enumerate(kqs) for _ in kq.selectors]
        asm = [int(var[bit0[iib[i] + k]]) for i, kq in enumerate(kqs) for k in kq.selectors]
        return {"kind": kind, "db": api.DeviceBatch(enc),
                "unit_inst": np.array(unit_inst, np.int32),
                "begin": np.arange(len(asm) + 1, dtype=np.int64), "asm": np.array(asm, np.int32)}
    if kind == "close":
        enc = B.scuba_encode_batch(irs_of(case, r))
        begin, asm = launch_constants(enc, r, int)
        db = api.DeviceBatch(enc)
        return {"kind": kind, "db": db, "begin": torch.from_numpy(begin).cuda(),
                "asm": torch.from_numpy(asm).cuda(),
                "values": torch.zeros(max(most_vars(case), db.total_vars), dtype=torch.uint8,
                                      device="cuda"),
                "conflict": torch.zeros(db.n, dtype=torch.uint8, device="cuda")}
    tr = make_trace(case, seed)
    return {"kind": kind, "trace": tr, "nodes": case["count"], "net": api.Mlp(seed=5),
            "grad": torch.zeros(B.SCUBA_MLP_NPARAM + 2, dtype=torch.float32, device="cuda"),
            "ds": torch.zeros(tr.max_rows, dtype=torch.float32, device="cuda")}


def run(state):
    kind = state["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "cdcl":
        return api.solve(state["db"], stats=False, search="cdcl", tuned=True,
                         time_budget_ms=TIME_MS)[0]
    if kind == "dpll":
        return api.solve(state["db"], stats=False, tuned=True, time_budget_ms=TIME_MS)[0]
    if kind == "learned":
        return api.solve(state["db"], stats=False, heuristic=B.SCUBA_HEUR_LEARNED,
                         mlp_weights=state["net"].weights, learned_depth=6,
                         time_budget_ms=TIME_MS)[0]
    if kind == "units":
        return api.solve_units(state["db"], state["unit_inst"], state["begin"], state["asm"],
                               search="cdcl", tuned=True, time_budget_ms=TIME_MS)[0]
    if kind == "close":
        rc = B._lib.scuba_propagate_batch(ctypes.byref(state["db"].struct()),
                                          state["begin"].data_ptr(), state["asm"].data_ptr(),
                                          state["values"].data_ptr(),
                                          state["conflict"].data_ptr(), stream)
        if rc != B.SCUBA_OK:
            raise RuntimeError("scuba_propagate_batch: %d" % rc)
        return state["values"], state["conflict"]
    rc = B._lib.scuba_mlp_grad(ctypes.byref(state["trace"].struct()), 0, state["nodes"],
                               state["net"].weights.data_ptr(), state["grad"].data_ptr(),
                               state["ds"].data_ptr(), stream)
    if rc != B.SCUBA_OK:
        raise RuntimeError("scuba_mlp_grad: %d" % rc)
    return state["grad"], state["ds"]


def work(case):
    kind, count = case["kind"], case["count"]
    if kind == "gradient":
        rows = int(node_rows(case, np.random.default_rng([0, 9])).sum())
        # features and targets in, score gradients out; forward, dW1, the hidden layer's gradient
        return {"bytes": rows * (2 * FEATURES + 8),
                "flops": rows * 2.0 * HIDDEN * (2 * FEATURES + 3)}
    # the formulas once (offsets, literals), verdicts or closures and models out
    r = np.random.default_rng([0, 3])
    if case["family"] == "3sat":
        clauses = int(round(4.26 * case["width"])) * count
        lits, nvars = 3 * clauses, case["width"] * count
    else:
        if kind == "units":
            irs = [frontend.kernel_queries(frontend.parse(stencil_text(r, case["width"])),
                                           bid_width=case["width"])[0].ir for _ in range(count)]
        else:
            irs = irs_of(case, r)
        enc = B.scuba_encode_batch(irs)
        clauses, lits, nvars = enc.total_clauses, enc.total_lits, enc.total_vars
    return {"bytes": 8.0 * clauses + 4.0 * lits + nvars + 21.0 * count, "flops": 0.0}


def exact(case, seed):
    if case["kind"] != "gradient":
        return None  # verdicts and closures are whole numbers
    s = prepare(case, seed)
    tr = s["trace"]
    w1, b1, w2, b2 = unpack(s["net"].weights)
    row, nrows, closed = (t.tolist() for t in (tr.node_row, tr.node_nrows, tr.node_closed))
    x_all = tr.x.view(torch.bfloat16).view(-1, FEATURES)
    grad = torch.zeros(B.SCUBA_MLP_NPARAM + 2, dtype=torch.float64, device="cuda")
    ds_all = torch.zeros(tr.max_rows, dtype=torch.float64, device="cuda")
    for k in range(case["count"]):
        rows = slice(row[k], row[k] + nrows[k])
        t = tr.target[rows].double()
        if not closed[k] or nrows[k] < 2 or float(t.sum()) <= 0:
            continue
        t = t / t.sum()
        x = x_all[rows].double()
        z = x @ w1 + b1
        h = torch.relu(z)
        logp = torch.log_softmax(h @ w2 + b2, 0)
        ds = torch.exp(logp) - t
        dh = torch.outer(ds, w2) * (z > 0)
        ds_all[rows] = ds
        grad += torch.cat([(x.T @ dh).reshape(-1), dh.sum(0), h.T @ ds, ds.sum().view(1),
                           -(t * logp).sum().view(1), torch.ones_like(ds[:1])])
    return grad, ds_all


def unpack(weights):
    """The packed device weights in 64 bits: W1 [16, 64], b1, w2, b2."""
    bf = weights[:2176].view(torch.bfloat16).double()
    fp = weights[2176:2436].view(torch.float32).double()
    return bf[:1024].view(HIDDEN, FEATURES).T, fp[:64], bf[1024:1088], fp[64]
