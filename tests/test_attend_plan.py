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
extern "C" int plan(int total, int units, int max_ch, int equal, int max_w, int may_merge, int pairs, int* workers, int* parts) {
  const AttendPlan p = rekv_attend_plan(total, units, max_ch, equal != 0, max_w, may_merge != 0, pairs != 0);
  *workers = p.workers;
  *parts = p.parts;
  return p.merge_inside;
}
extern "C" int merge_ahead(int parts, int blocks, int sms) { return rekv_merge_ahead(parts, blocks, sms); }
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
        w, parts = ctypes.c_int(), ctypes.c_int()
        inside = fn(sum(chunks) * lh, len(chunks) * lh, max(chunks), int(min(chunks) == max(chunks)), max_w, int(may_merge),
                    int(max_w <= 74), ctypes.byref(w), ctypes.byref(parts))
        return w.value, bool(inside), parts.value
    return call


def _parts(chunks, lh, workers):
    """the parts of every unit"""
    total, at = sum(chunks) * lh, 0
    for n in chunks * min(lh, 64):
        yield (at + n - 1) * workers // total - at * workers // total + 1
        at += n


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
            w, _, _ = plan(chunks, lh, max_w, may_merge)
            assert 1 <= w <= min(max_w, sum(chunks) * lh), (chunks, lh, max_w, may_merge, w)


def test_units_joined_in_the_kernel_have_at_most_four_parts(plan):
    for chunks, lh, max_w in _batches(4000):
        for may_merge in (True, False):
            w, inside, _ = plan(chunks, lh, max_w, may_merge)
            assert inside or may_merge
            if not inside:
                continue
            assert max(_parts(chunks, lh, w)) <= 4, (chunks, lh, max_w, may_merge, w)


def test_parts_of_a_unit_are_known(plan):
    """The most parts that a unit has: a bound, and for equal units the number itself."""
    for chunks, lh, max_w in _batches(4000):
        w, _, parts = plan(chunks, lh, max_w, True)
        most = max(_parts(chunks, lh, w))
        assert most <= parts, (chunks, lh, max_w, w)
        if min(chunks) == max(chunks) and len(chunks) * lh <= w and w % (len(chunks) * lh) == 0:
            assert most == parts, (chunks, lh, max_w, w)


def test_the_gpu_tests_of_the_merge_launch_reach_what_they_name(plan, rules):
    """One layer of test_parity_gpu.py's shapes (7 query heads per KV head, 196 tokens per frame at a pitch of 200, two trailing
    frames) on 148 SMs: the parts of a unit, and the parts in flight."""
    from tests.test_parity_gpu import MERGED
    earlier = [(1, [20], 31, 18, 10), (2, [37], 31, 18, 10), (3, [20], 31, 18, 10), (4, [20], 31, 18, 10), (5, [9], 31, 18, 10),
               (6, [40], 31, 6, 4), (8, [20], 31, 9, 4), (8, [5], 31, 18, 10)]
    seen = set()
    for Hkv, lengths, k, parts, ahead in MERGED + earlier:
        rows = [7 * n for n in lengths]
        pairs = max(rows) > 128
        units = sum(-(-r // (256 if pairs else 128)) for r in rows)
        chunks = -(-((k + 1) * 200 + 196) // 128)
        w, inside, p = plan([chunks] * units, Hkv, 74 if pairs else 148, True)
        assert not inside and p == parts == max(_parts([chunks] * units, Hkv, w))
        assert rules.merge_ahead(p, 32 * Hkv * sum(-(-r // 128) for r in rows), 148) == ahead
        seen.add((pairs, ahead, -(-parts // (2 * ahead)) > 1))
    assert {(pairs, ahead) for pairs, ahead, _ in seen} == {(pairs, ahead) for pairs in (False, True) for ahead in (4, 8, 10)}
    assert (True, 8, True) in seen and (False, 4, True) in seen   # (several rounds)


@pytest.mark.parametrize("layers,n_tokens,expected", [(20, 16, True), (20, 80, False), (10, 80, False), (4, 16, False)])
def test_output_warps_only_on_single_ctas_of_several_long_segments(plan, rules, layers, n_tokens, expected):
    """The units of test_parity_gpu.py's and test_failure_paths_gpu.py's launches of several segments: 8 KV heads of two query heads
    and 34 chunks; 16 tokens are 32 rows (single CTAs), 80 are 160 (pairs).  (4 layers: a worker for every unit.)"""
    pairs = n_tokens * 2 > 128
    workers, _, _ = plan([34], 8 * layers, 74 if pairs else 148, True)
    assert rules.output_warps(workers, 8 * layers, 34, int(pairs)) == int(expected)
    assert rules.output_warps(workers, 8 * layers, 31, int(pairs)) == 0
