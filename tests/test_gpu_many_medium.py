"""Batches with more units than one block on every SM has warps, whose largest
instance leaves no room for two blocks with positions and marks in shared memory, and
batches with a budget, which take two blocks of 8 warps: the verdicts of the DPLL
search, and models that verify, on both sides of each line."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from raw_cnf import model_ok, solve_raw
from test_gpu_launch_shapes import sat_instances
from test_gpu_prep_shapes import libs  # noqa: F401

pytestmark = pytest.mark.gpu


def padded(cnf, n):
    """The instance among n variables, the added ones in an implication chain."""
    m, cls = cnf
    return n, cls + [[-v, v + 1] for v in range(m + 1, n)]


@pytest.mark.parametrize("vmax", [1800, 1900, 3100, 3300, 4905])
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("budget", [0, 1 << 30])
def test_placement_by_batch_size(libs, vmax, extra, budget):
    api, _ = libs
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    kinds = sat_instances(40, 20, 70)
    kinds[7] = padded(kinds[7], vmax)
    count = (12 if budget else 8) * sms + extra
    cnfs = [kinds[i % 40] if i % 40 != 7 or i < 400 else kinds[8] for i in range(count)]
    _, ref, _, _, _ = solve_raw(api, kinds, search="dpll", time_budget_ms=30000)
    want = np.array([ref[i % 40] if i % 40 != 7 or i < 400 else ref[8] for i in range(count)])
    st, v, m, vb, _ = solve_raw(api, cnfs, search="cdcl", time_budget_ms=60000,
                                decision_budget=budget)
    assert st == 0 and (v == want).all() and set(ref.tolist()) == {0, 1}
    assert all(model_ok(cnfs[i][1], m, vb[i]) for i in np.flatnonzero(v == 1))
