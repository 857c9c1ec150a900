"""The searches' arithmetic that needs no GPU (csrc/rules.h), compiled here."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r'''
#include "rules.h"
extern "C" uint64_t elapsed_ns(uint64_t a, uint64_t b) { return scuba::elapsed_ns(a, b); }
extern "C" uint32_t flush_steps(uint64_t e, uint64_t l, uint64_t v) {
  return scuba::flush_steps(e, l, v);
}
'''


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I",
                           os.path.join(ROOT, "paper_2601_21552_gb300", "csrc"),
                           str(d / "r.cpp"), "-o", str(d / "r.so")])
    return ctypes.CDLL(str(d / "r.so"))


@pytest.mark.parametrize("start,now,want", [
    (1000, 1000, 0), (1000, 1001, 1), (1000, 999, 0), (5_000_000, 1, 0),
    (1, 600_000_000_001, 600_000_000_000), (2**63 - 5, 2**63 + 5, 10), (2**63 + 5, 2**63 - 5, 0),
    (2**64 - 3, 4, 7)])
def test_a_clock_behind_the_start_reads_zero(rules, start, now, want):
    rules.elapsed_ns.argtypes = [ctypes.c_uint64] * 2
    rules.elapsed_ns.restype = ctypes.c_uint64
    assert rules.elapsed_ns(start, now) == want


@pytest.mark.parametrize("entries,words,variables", [
    (0, 0, 0), (30_000, 1 << 18, 2000), ((1 << 26) - 1, 0, 0), (1 << 26, 0, 0),
    (60_000_000, 1 << 24, 900_000), (1 << 27, 0, 0), (1 << 31, 0, 0), ((1 << 32) - 1, 0, 0),
    ((1 << 32) - 1, 1 << 30, 1 << 29)])
def test_counters_cannot_wrap_between_flushes(rules, entries, words, variables):
    rules.flush_steps.argtypes = [ctypes.c_uint64] * 3
    rules.flush_steps.restype = ctypes.c_uint32
    steps, most = rules.flush_steps(entries, words, variables), entries + words + variables
    assert steps in (1, 2, 4, 8, 16, 32, 64)
    assert steps * most < 2**32 or steps == 1
    assert steps == 64 or 2 * steps * most >= 2**32   # no oftener than it has to be
