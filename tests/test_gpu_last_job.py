"""The verdict that the last open job of an instance writes: instances cut into
subtrees or cubes as early as the options allow, whose jobs end all at once --
with a model, without one, or out of budget. A model found or a budget reached in
any of them is never lost to the last one's UNSAT."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from raw_cnf import model_ok, solve_raw
from test_gpu_launch_shapes import sat_instances
from test_gpu_prep_shapes import libs  # noqa: F401

pytestmark = pytest.mark.gpu

EAGER = {"dpll": dict(split_min=1, split_interval=1),
         "cdcl": dict(split_min=1, split_interval=1, restart_unit=1)}


@pytest.mark.parametrize("search", ["dpll", "cdcl"])
@pytest.mark.parametrize("budget", [0, 300])
def test_no_result_is_lost_among_many_jobs(libs, search, budget):
    api, _ = libs
    cnfs = sat_instances(40, 60, 100)
    st, ref, _, _, _ = solve_raw(api, cnfs, search=search, split=False)
    assert st == 0 and set(ref.tolist()) == {0, 1}
    unknown = 0
    for _ in range(25):
        st, v, m, vb, _ = solve_raw(api, cnfs, search=search, decision_budget=budget,
                                    **EAGER[search])
        assert st == 0
        unknown += int((v == 2).sum())
        assert (v == ref)[v != 2].all()
        assert all(model_ok(cnfs[i][1], m, vb[i]) for i in np.flatnonzero(v == 1))
    assert (unknown > 0) == (budget > 0)
