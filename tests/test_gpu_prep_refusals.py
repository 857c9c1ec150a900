"""A refused clause range among thousands of instances: the block that meets it
ends the whole call while others start, work and finish. Every entry point
reports SCUBA_ERR_MALFORMED, no verdict is given, and the next well-formed
batch is answered."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from raw_cnf import pack, solve_raw
from test_gpu_prep_shapes import libs  # noqa: F401

pytestmark = pytest.mark.gpu

N = 6000


def batch(large):
    """N small satisfiable instances, with `large` one of 4,000 variables among
    them (blocks of 32 warps, instances cut into ranges)."""
    cnfs = [(20, [[-v, v + 1] for v in range(1, 20)] + [[1, 5, -9, 7]] * 20)] * N
    if large:
        cnfs[N // 3] = (4000, [[-v, v + 1] for v in range(1, 4000)])
    return cnfs


@pytest.mark.parametrize("large", [False, True], ids=["small", "ranges"])
@pytest.mark.parametrize("at", [1, 700, N // 2, N - 1])
def test_malformed_range_among_thousands(libs, large, at):
    api, B = libs
    cnfs = batch(large)
    icb, cb, lits, nv, vb, L = pack(cnfs)
    icb[at] += 50 + (icb[at + 1] - icb[at])   # past the next instance's first clause
    t = lambda a: torch.from_numpy(a).cuda()
    keep = [t(x) for x in (icb, cb, lits, nv, vb)]
    b = B.make_batch(N, int(nv.max()), len(cb) - 1, L, int(vb[-1]),
                     *(x.data_ptr() for x in keep))
    verdict = torch.empty(N, dtype=torch.uint8, device="cuda")
    model = torch.zeros(int(vb[-1]), dtype=torch.uint8, device="cuda")
    values, conflict = torch.zeros_like(model), torch.zeros_like(verdict)
    none = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    for _ in range(10):
        for search in ("dpll", "cdcl"):
            verdict.fill_(9)
            B.scuba_solve_batch_ex(b, verdict.data_ptr(), model.data_ptr(), s,
                                   api.options(search=search, time_budget_ms=20000))
            assert B.scuba_sync_status(s) == B.SCUBA_ERR_MALFORMED
            assert bool((verdict == 2).all())
        assert B._lib.scuba_propagate_batch(b, none.data_ptr(), keep[2].data_ptr(),
                                            values.data_ptr(), conflict.data_ptr(), s) == 0
        assert B.scuba_sync_status(s) == B.SCUBA_ERR_MALFORMED
    st, v, _, _, _ = solve_raw(api, cnfs)
    assert st == 0 and (v == 1).all()
