"""The rule that deals a launch's chunks to the workers of the tensor-core attention kernel (csrc/attend_plan.h, plain host
code), walked over batches of equal and very unequal units: no worker is left without a chunk -- it would read the queries of
a unit beyond the last, and be counted as a part that nobody writes -- and no unit whose parts the kernel joins itself has more
than the four it can join."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_00540_b200", "csrc")
SOURCE = """
#include "attend_plan.h"
extern "C" int plan(int total, int units, int max_ch, int equal, int max_w, int may_merge, int pairs, int* workers) {
  const AttendPlan p = rekv_attend_plan(total, units, max_ch, equal != 0, max_w, may_merge != 0, pairs != 0);
  *workers = p.workers;
  return p.merge_inside;
}
extern "C" int output_warps(int workers, int units, int max_ch, int pairs) {
  return rekv_attend_output_warps(workers, units, max_ch, pairs != 0);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(src)])
    return ctypes.CDLL(str(so))


@pytest.fixture(scope="module")
def plan(rules):
    fn = rules.plan

    def call(chunks, lh, max_w, may_merge):
        """chunks: of one (layer, KV head)'s units, in launch order; lh: how many (layer, KV head) there are"""
        w = ctypes.c_int()
        inside = fn(sum(chunks) * lh, len(chunks) * lh, max(chunks), int(min(chunks) == max(chunks)), max_w, int(may_merge),
                    int(max_w <= 74), ctypes.byref(w))
        return w.value, bool(inside)
    return call


def _batches(n):
    """unit lengths as batches make them: questions of one to four row blocks over a shared context, X's lengths equal, near,
    or with one very long one among short ones"""
    rng = random.Random(2503)
    for _ in range(n):
        context = rng.choice([0, 1, 2, 3, 7, 15, 40, 113])
        chunks = []
        style = rng.choice(["equal", "near", "one long", "any"])
        nq = rng.randint(1, 16)
        for i in range(nq):
            x = {"equal": 1, "near": rng.randint(0, 2), "one long": 1, "any": rng.randint(0, 64)}[style]
            if style == "one long" and i == nq // 2:
                x = rng.choice([4, 10, 20, 69, 200])
            chunks += [max(1, context + x)] * rng.randint(1, 4)
        yield chunks, rng.choice([1, 2, 4, 8, 16, 28 * 4, 80 * 8]), rng.choice([1, 2, 66, 74, 132, 148])
    for chunks, lh, max_w in ([1, 1, 10], 1, 74), ([2, 2, 10], 4, 74), ([2, 2, 2, 20], 4, 148), ([7] * 4 + [69], 32, 148), \
            ([15] * 7 + [200], 16, 148):
        yield chunks, lh, max_w


def test_every_worker_has_a_chunk(plan):
    for chunks, lh, max_w in _batches(4000):
        for may_merge in (True, False):
            w, _ = plan(chunks, lh, max_w, may_merge)
            assert 1 <= w <= min(max_w, sum(chunks) * lh), (chunks, lh, max_w, may_merge, w)


def test_units_joined_in_the_kernel_have_at_most_four_parts(plan):
    for chunks, lh, max_w in _batches(4000):
        total = sum(chunks) * lh
        for may_merge in (True, False):
            w, inside = plan(chunks, lh, max_w, may_merge)
            assert inside or may_merge
            if not inside:
                continue
            at = 0
            for n in chunks * min(lh, 64):
                parts = (at + n - 1) * w // total - at * w // total + 1
                assert parts <= 4, (chunks, lh, max_w, may_merge, w)
                at += n


@pytest.mark.parametrize("layers,n_tokens,expected", [(20, 16, True), (20, 80, False), (10, 80, False), (4, 16, False)])
def test_output_warps_only_on_single_ctas_of_several_long_segments(plan, rules, layers, n_tokens, expected):
    """The units of test_parity_gpu.py's and test_failure_paths_gpu.py's launches of several segments: 8 KV heads of two query heads
    and 34 chunks; 16 tokens are 32 rows (single CTAs), 80 are 160 (pairs).  (4 layers: a worker for every unit.)"""
    pairs = n_tokens * 2 > 128
    workers, _ = plan([34], 8 * layers, 74 if pairs else 148, True)
    assert rules.output_warps(workers, 8 * layers, 34, int(pairs)) == int(expected)
    assert rules.output_warps(workers, 8 * layers, 31, int(pairs)) == 0
