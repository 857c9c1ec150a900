"""Propagation rounds that assign many literals at once: one decision falsifies a
literal with k binary clauses, so up to 32 lanes append to the trail in one
step, more than the ring of recent literals holds. The next round has to see
every one of them: a pair of the implied literals excludes itself, so that the
first branch (the lowest variable false) must fail whatever the pair. Exact
verdicts, and models that satisfy every clause."""
import pytest

torch = pytest.importorskip("torch")

from raw_cnf import model_ok, solve_raw

pytestmark = pytest.mark.gpu


def fan(k, a, b, unsat):
    """Variable 1, k implied ones (2 .. k+1), one more that makes variable 1's
    true branch fail as well if unsat."""
    cls = [[1, i + 2] for i in range(k)] + [[-(a + 2), -(b + 2)]]
    if unsat:
        cls += [[-1, k + 2], [-1, -(k + 2)]]
    return k + 2, cls


@pytest.mark.parametrize("search", ["dpll", "cdcl"])
@pytest.mark.parametrize("k", [2, 15, 16, 17, 18, 31, 32, 33, 47, 64, 100])
def test_every_literal_of_a_wide_round_is_propagated(search, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_21552_gb300 import build
    build.build()
    from paper_2601_21552_gb300 import api
    pairs = [(a, b) for a in range(k) for b in range(a + 1, k)]
    pairs = pairs[:: max(1, len(pairs) // 300)] + [(0, k - 1), (k - 2, k - 1)]
    cnfs = [fan(k, a, b, unsat) for a, b in pairs for unsat in (False, True)]
    st, v, m, vb, _ = solve_raw(api, cnfs, search=search, time_budget_ms=30000)
    assert st == 0
    for i, (_, cls) in enumerate(cnfs):
        assert v[i] == (0 if i % 2 else 1), (k, pairs[i // 2], i % 2)
        assert i % 2 or model_ok(cls, m, vb[i]), (k, pairs[i // 2])
