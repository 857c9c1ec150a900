"""Results do not depend on the launch shape that a rule or an option picks:
clause learning with 1 to 8 warps a block and one or two blocks an SM, learned
branching on batches just below and above a unit for every warp of its large
shape, and the closure of a conflicting instance, which blocks of several warps
share when there are few instances and one warp propagates when there are many
-- its values are those of the fixed order either way."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from raw_cnf import model_ok, solve_raw
from test_gpu_prep_shapes import closure, libs  # noqa: F401

pytestmark = pytest.mark.gpu


def sat_instances(count, lo, hi):
    from workloads import queries
    out = []
    for s in range(count):
        n, l = queries.random_3sat(9100 + s, lo, hi)
        out.append((n, [list(map(int, c)) for c in l]))
    return out


@pytest.mark.parametrize("wpb,bps", [(1, 1), (1, 2), (5, 2), (6, 1), (6, 2), (7, 2), (8, 1),
                                     (8, 2), (0, 0)])
def test_clause_learning_shapes(libs, wpb, bps):
    api, _ = libs
    cnfs = sat_instances(48, 40, 90)
    _, ref, _, _, _ = solve_raw(api, cnfs, search="dpll", time_budget_ms=30000)
    st, v, m, vb, _ = solve_raw(api, cnfs, search="cdcl", time_budget_ms=30000,
                                warps_per_block=wpb, blocks_per_sm=bps)
    assert st == 0 and v.tolist() == ref.tolist() and set(ref.tolist()) == {0, 1}
    assert all(model_ok(cnfs[i][1], m, vb[i]) for i in range(len(cnfs)) if v[i] == 1)


@pytest.mark.parametrize("extra", [-1, 0])
def test_learned_branching_around_the_large_shape(libs, extra):
    api, B = libs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cnfs = sat_instances(64, 12, 40)
    cnfs = [cnfs[i % 64] for i in range(24 * sms + extra)]
    net = api.Mlp(seed=2)
    st, v, m, vb, _ = solve_raw(api, cnfs, heuristic=B.SCUBA_HEUR_LEARNED, learned_depth=6,
                                mlp_weights=net.weights, time_budget_ms=30000)
    _, ref, _, _, _ = solve_raw(api, cnfs[:64], search="cdcl", time_budget_ms=30000)
    assert st == 0 and v.tolist() == [int(ref[i % 64]) for i in range(len(cnfs))]
    assert all(model_ok(cnfs[i][1], m, vb[i]) for i in range(len(cnfs)) if v[i] == 1)


@pytest.mark.parametrize("n", [2048, 5000, 17000])
def test_conflicting_closure_alone_and_among_many(libs, n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(n)
    order = [1] + (rng.permutation(n - 1) + 2).tolist()
    cls = [[-order[int(rng.integers(0, i))], order[i]] for i in range(1, n)]   # a random tree
    cls += [[-order[n // 2], -order[n - 1]], [-order[n // 3], -order[n - 2]]]
    rng.shuffle(cls)
    alone, c1, _ = closure(libs, [(n, cls)], [[1]])
    small = [(3, [[-1, 2], [-2, 3]])] * (24 * sms)
    many, c2, vb = closure(libs, [(n, cls)] + small, [[1]] + [[1]] * len(small))
    assert c1[0] == 1 and c2[0] == 1
    assert np.array_equal(alone, many[:n])
    assert not c2[1:].any()
    assert len(set(map(bytes, many[n:].reshape(-1, 3)))) == 1  # the small ones agree
