"""Occurrence lists longer than a 16-bit count: of a literal that one warp of the
preparation alone meets more than 65,535 times (long clauses that repeat it, side
by side), or that only all warps of the block together do; the literal in the low
or the high half of its counter word, the instance whole or cut into literal
ranges. The closures equal the CPU's, every time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_bcp import cpu_closure
from test_gpu_prep_shapes import closure, libs  # noqa: F401

pytestmark = pytest.mark.gpu


def clauses(nvars, sign, spread):
    """65,536 or more occurrences of literal `sign`, which the closure falsifies."""
    rng = np.random.default_rng(nvars + sign + 7 * spread)
    ys = rng.integers(2, nvars + 1, 1100).tolist()
    heavy = [[sign] * 61 + [y] for y in ys]                   # 67,100 occurrences
    light = [[-sign, int(y)] for y in rng.integers(2, nvars + 1, 40 * 1100)]
    cls = light[:16 * 1100] + heavy + light[16 * 1100:]
    if spread:
        rng.shuffle(cls)
    cls.insert(9, [2])
    return cls + [[-2, -3, 4], [sign, 5, 5]]


@pytest.mark.parametrize("nvars", [200, 4000], ids=["whole", "ranges"])
@pytest.mark.parametrize("sign", [1, -1], ids=["low", "high"])
@pytest.mark.parametrize("spread", [0, 1], ids=["one_warp", "all_warps"])
def test_closure_with_long_lists(libs, nvars, sign, spread):
    cls = clauses(nvars, sign, spread)
    want_c, want_v = cpu_closure(nvars, cls, [-sign])
    assert not want_c and (want_v != 0).sum() > 190   # every y follows
    small = (3, [[1], [-1, 2]])
    for _ in range(20):
        values, conflict, vb = closure(libs, [small, (nvars, cls), small], [[], [-sign], [3]])
        assert not conflict.any()
        assert (values[3:3 + nvars] == want_v).all()
        assert values[:3].tolist() == [1, 1, 0] and values[3 + nvars:].tolist() == [1, 1, 1]
