"""The occurrence lists that the preparation builds, seen through the closure of
unit propagation: CNFs at the edges of its tiles and ranges -- a batch whose
literals just fit the small blocks' counters and one that does not, instances
cut into several literal ranges, empty instances among others, clauses of one
to many literals with duplicates and tautologies, a literal that occurs more
than 65,535 times -- against a plain CPU closure; malformed headers are
refused as before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from raw_cnf import pack, solve_raw
from test_gpu_bcp import cpu_closure

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def libs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_21552_gb300 import build
    build.build()
    from paper_2601_21552_gb300 import api, binding
    return api, binding


def chain(n, extra, rng):
    """Implication chain over all n variables (assuming 1 assigns them all),
    mixed with clauses that stay open or satisfied."""
    order = rng.permutation(np.arange(2, n + 1))
    sign = np.where(rng.random(n + 1) < 0.5, 1, -1)
    cls, prev = [], 1
    for v in order:
        lit = int(sign[v] * v)
        cls.append([-prev, lit] if rng.random() < 0.5 else [lit, -prev, -prev])
        prev = lit
    for _ in range(extra):
        k = int(rng.integers(1, 6))
        c = [int(sign[v] * v) for v in rng.integers(2, n + 1, k)]
        c += [int(rng.integers(1, n + 1)) * (1 if rng.random() < 0.5 else -1)]
        cls.append(c + [int(sign[x] * x) if x > 1 else 1 for x in [int(rng.integers(1, n + 1))]])
    cls.append([5, -5, 3])
    rng.shuffle(cls)
    return n, cls


def closure(libs, cnfs, assumptions):
    api, B = libs
    icb, cb, lits, nv, vb, _ = pack(cnfs)
    db = api.DeviceBatch.from_csr(icb, cb, lits, nv, vb)
    ab = np.concatenate([[0], np.cumsum([len(a) for a in assumptions])]).astype(np.int64)
    al = np.array([x for a in assumptions for x in a] or [0], np.int32)
    d_ab, d_al = torch.from_numpy(ab).cuda(), torch.from_numpy(al).cuda()
    values = torch.full((max(int(vb[-1]), 1),), 7, dtype=torch.uint8, device="cuda")
    conflict = torch.full((len(cnfs),), 7, dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    assert B._lib.scuba_propagate_batch(db.struct(), d_ab.data_ptr(), d_al.data_ptr(),
                                        values.data_ptr(), conflict.data_ptr(), s) == 0
    assert B.scuba_sync_status(s) == 0
    return values.cpu().numpy(), conflict.cpu().numpy(), vb


@pytest.mark.parametrize("sizes", [
    [1843, 5, 1, 700], [1844, 40, 3], [3264, 1632, 1633, 9], [5000, 4896, 17],
    [33, 64, 31, 32, 65] * 60], ids=["fits8", "over8", "ranges2", "ranges4", "many"])
def test_closure_over_block_and_range_edges(libs, sizes):
    rng = np.random.default_rng(sum(sizes))
    cnfs, asm = [], []
    for n in sizes:
        cnfs.append(chain(n, 3 * n, rng) if n >= 5 else (n, [[1], [-1, n]]))
        asm.append([1] if n >= 5 and rng.random() < 0.8 else [])
        cnfs.append((3, []))   # an instance without clauses
        asm.append([2])
    values, conflict, vb = closure(libs, cnfs, asm)
    for i, (n, cls) in enumerate(cnfs):
        if not cls:   # the CPU closure wants a clause
            assert conflict[i] == 0 and values[vb[i]:vb[i] + n].tolist() == [0, 1, 0]
            continue
        want_c, want_v = cpu_closure(n, [c for c in cls if not any(-x in c for x in c)], asm[i])
        assert bool(conflict[i]) == want_c, i
        if not want_c:
            assert (values[vb[i]:vb[i] + n] == want_v).all(), i


@pytest.mark.parametrize("nvars", [200, 4000], ids=["small", "ranges"])
def test_literal_with_more_than_65535_occurrences(libs, nvars):
    rng = np.random.default_rng(3)
    ys = rng.integers(2, nvars + 1, 70000)
    cls = [[-1, int(y)] for y in ys] + [[-2, -3, nvars], [4], [-4, 6, 5, 6, 7]]
    cls[12345], cls[-2] = cls[-2], cls[12345]   # the unit clause inside the run
    values, conflict, vb = closure(libs, [(nvars, cls), (2, [[1], [-1, 2]])], [[1], []])
    want_c, want_v = cpu_closure(nvars, cls, [1])
    assert not want_c and not conflict.any()
    assert (values[:nvars] == want_v).all()
    assert values[nvars:].tolist() == [1, 1]


def test_entries_are_complete_and_units_in_order(libs):
    """Every literal of a clause finds it: falsify all but one literal of each
    clause of every length, the last one must follow."""
    rng = np.random.default_rng(8)
    cnfs, asm, want = [], [], []
    for n in list(range(2, 9)) + [40]:
        c = [int(v) * (1 if rng.random() < 0.5 else -1) for v in rng.permutation(n) + 1]
        for k in range(n):
            cnfs.append((n + 2, [c, [n + 1], [n + 1, n + 2], [-n - 2]]))
            asm.append([-x for j, x in enumerate(c) if j != k])
            want.append((abs(c[k]) - 1, 1 if c[k] > 0 else 2))
    values, conflict, vb = closure(libs, cnfs, asm)
    assert not conflict.any()
    for i, (v, x) in enumerate(want):
        n = cnfs[i][0]
        assert values[vb[i] + v] == x and values[vb[i] + n - 2] == 1 and values[vb[i] + n - 1] == 2


@pytest.mark.parametrize("where", ["first", "last", "order", "beyond", "clause"])
def test_malformed_offsets_are_refused(libs, where):
    api, B = libs
    icb, cb, lits, nv, vb, L = pack([(3, [[1, 2], [3]]), (2, [[-1, 2], [1]]), (1, [[1]])])
    if where == "first": icb[0] = 1
    if where == "last": icb[-1] -= 1
    if where == "order": icb[1], icb[2] = icb[2], icb[1]
    if where == "beyond": icb[1] = 99
    if where == "clause": cb[1] = L + 5
    t = lambda a: torch.from_numpy(a).cuda()
    keep = [t(x) for x in (icb, cb, lits, nv, vb)]
    b = B.make_batch(3, 3, len(cb) - 1, L, int(vb[-1]), *(x.data_ptr() for x in keep))
    verdict = torch.full((3,), 9, dtype=torch.uint8, device="cuda")
    model = torch.zeros(6, dtype=torch.uint8, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for search in ("dpll", "cdcl"):
        B.scuba_solve_batch_ex(b, verdict.data_ptr(), model.data_ptr(), s,
                               api.options(search=search, time_budget_ms=20000))
        assert B.scuba_sync_status(s) == B.SCUBA_ERR_MALFORMED
        v = verdict.cpu().numpy()
        assert v[0] == 2 if where == "clause" else (v == 2).all()


def test_verdicts_of_large_and_small_instances_together(libs):
    api, B = libs
    rng = np.random.default_rng(21)
    cnfs = [chain(4000, 4000, rng), (3, [[1], [-1, 2], [-2]]), chain(900, 900, rng), (2, []), (1, [[]])]
    for search in ("dpll", "cdcl"):
        st, v, m, vb, _ = solve_raw(api, cnfs, search=search)
        assert st == 0
        assert v.tolist() == [1, 0, 1, 1, 0]
        for i in (0, 2):
            assert all(any((m[vb[i] + abs(x) - 1] == 1) == (x > 0) for x in c) for c in cnfs[i][1])
