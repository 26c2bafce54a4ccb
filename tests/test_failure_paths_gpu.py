"""The device-side failure path: a bounded wait that runs out.

Every wait inside the attention kernels (on a tile copy, a matrix product, another warp) has an iteration limit;
when it is reached the kernel writes REKV_ERR_TIMEOUT to the status word, waits (again bounded) for its own copies
in flight, releases tensor memory and returns, so the context stays usable.  The test-only call
rekv_test_set_wait_limit shortens the limit and makes the copy producer of one CTA leave out one tile copy, so
that the wait for that tile expires with nothing in flight -- no fault, no trap, no endless loop.  Checked: the
call returns, rekv_check_status reports REKV_ERR_TIMEOUT exactly once, and the next question on the same context
matches the oracle.
"""
import pytest
import torch

from paper_2503_00540_b200 import rekv
from tests import harness as H

pytestmark = pytest.mark.gpu


def _expire_then_recover(s: H.Shape, lengths, skip_entry: int):
    g = H.build_gpu(s, max_questions=len(lengths), max_q_tokens=sum(lengths))
    o = H.build_oracle(s)
    q, cu = H.questions(s, lengths, device="cuda")
    # 1. a healthy question first: the kernels' function attributes and the context are set up
    out0 = g.question(q, cu, s.k, s.T)
    g.check_status()
    # 2. the wait runs out
    g.test_set_wait_limit(20000, skip_entry)
    g.question(q, cu, s.k, s.T)
    with pytest.raises(rekv.RekvError) as e:
        g.check_status()
    assert e.value.code == rekv.ERR_TIMEOUT and "wait expired" in str(e.value)
    g.check_status()  # the status word was cleared by the read
    # 3. the same context answers the next question correctly
    g.test_set_wait_limit(0, -1)
    out1 = g.question(q, cu, s.k, s.T)
    g.check_status()
    assert torch.equal(out0, out1)
    for i in range(len(lengths)):
        ref = o.question(q[:, cu[i]:cu[i + 1]].cpu().contiguous(), s.k, s.T)
        H.assert_attention(out1[:, cu[i]:cu[i + 1]], ref["out"], f"after the expired wait, question {i}")
    g.close()


@pytest.mark.parametrize("skip_entry", [0, 1, 3])
def test_tensor_core_kernel_gives_up_when_a_tile_never_arrives(skip_entry):
    """64 query rows per KV head: the tcgen05 kernel.  Entry 0 is a K tile (the S product waits for it), entry 1 a V
    tile (the P V product waits), entry 3 the second chunk's V tile of the first CTA's range (eight units
    of 15 chunks, eight CTAs each)."""
    s = H.Shape(L=4, Hq=8, Hkv=2, Nf=48, T=60, W=4, k=36, seed=7)
    _expire_then_recover(s, [16], skip_entry)


def test_a_cta_that_gives_up_leaves_its_units_unfinished_and_their_counters_are_cleared():
    """80 units of two row tiles, most of them cut in two parts that the attention kernel joins itself by counting
    the parts per unit.  The first CTA gives up on its first K tile: its parts are never counted, the units it shares
    stay unfinished behind the status word, and reading the status clears the counters -- the next question would
    otherwise join the wrong parts."""
    s = H.Shape(L=10, Hq=16, Hkv=8, Nf=100, T=28, W=4, k=16, seed=2503)
    _expire_then_recover(s, [80], 0)


def test_decode_kernel_gives_up_when_a_frame_never_arrives():
    """One query token (4 rows per KV head): the load-bound decode kernel."""
    s = H.Shape(L=4, Hq=8, Hkv=2, Nf=48, T=60, W=4, k=36, seed=7)
    _expire_then_recover(s, [1], 0)


@pytest.mark.parametrize("n_tokens,skip_entry", [(16, 0), (16, 1), (16, 68), (16, 69), (80, 0), (80, 1), (80, 69), (80, 136)])
def test_results_of_several_segments_are_given_up_with_the_rest(n_tokens, skip_entry):
    """160 units of 34 chunks over 144 single CTAs (16 tokens) or 64 pairs (80), several segments each.  The first CTA misses its
    first K tile, its first V tile, or one of its second or third segment (34 chunks each): the warps that put out a segment's
    result then wait for a product that never comes, and where they are warps of their own the softmax warps wait for them.  A
    pair's CTAs leave together."""
    s = H.Shape(L=20, Hq=16, Hkv=8, Nf=80, T=56, W=2, k=52, seed=7)
    _expire_then_recover(s, [n_tokens], skip_entry)


@pytest.mark.parametrize("s,nq,ns,skip_entry", [
    (H.Shape(L=3, Hq=28, Hkv=4, Nf=196, T=80, W=2, k=70, seed=7), 1, 48, 0),    # two frames on a CTA, the first missing
    (H.Shape(L=3, Hq=28, Hkv=4, Nf=196, T=80, W=2, k=70, seed=7), 1, 48, 1),    # ... the second
    (H.Shape(L=2, Hq=32, Hkv=8, Nf=16, T=10, W=2, k=6, seed=7), 16, 5, 0),      # eight frames in a step, X's copies behind them
], ids=["first", "second", "x_in_flight"])
def test_a_frame_rotated_before_the_dependency_wait_never_arrives(s, nq, ns, skip_entry):
    """One token at a time over a context that earlier launches on the stream have read: its first frames are copied, and their keys
    rotated, before the dependency wait.  The wait for the frame that is left out is the rotation's."""
    g = H.build_gpu(s, max_questions=nq, max_q_tokens=nq, max_self_tokens=nq * ns, rope_theta=1e6)
    q, cu = H.questions(s, [1] * nq, device="cuda")
    ks, vs, cus = H.self_kv(s, [ns] * nq, device="cuda")
    g.gather(g.retrieve(q, cu, s.k, s.T)[0], nq, s.k, s.T)

    def token():
        return torch.stack([g.attend_full_layer(l, q[l], ks[l], vs[l], cu, cus) for l in range(s.L)])
    token()
    out0 = token()
    g.check_status()
    g.test_set_wait_limit(20000, skip_entry)
    token()
    with pytest.raises(rekv.RekvError) as e:
        g.check_status()
    assert e.value.code == rekv.ERR_TIMEOUT
    g.check_status()
    g.test_set_wait_limit(0, -1)
    assert torch.equal(token(), out0)
    assert torch.equal(token(), out0)
    g.check_status()
    g.close()


@pytest.mark.parametrize("L,lengths", [(1, [16]), (12, [5, 3, 4])])  # clusters of 16 and of 8 CTAs
@pytest.mark.parametrize("mode", [rekv.TEST_RETRIEVE_SKIP_SUM, rekv.TEST_RETRIEVE_SKIP_SCORE])
def test_one_launch_retrieval_gives_up_when_a_part_never_arrives(L, lengths, mode):
    """A CTA of the first layer's cluster leaves out its part of the question vectors (every CTA of the cluster waits for it)
    or a score (the CTA that selects waits): the launch returns, the layer's list is empty and its context table safe to
    follow, and the next question is answered as before."""
    s = H.Shape(L=L, Hq=8, Hkv=2, Nf=16, T=60, W=4, k=8, seed=7)
    g = H.build_gpu(s, max_questions=len(lengths), max_q_tokens=sum(lengths))
    q, cu = H.questions(s, lengths, device="cuda")
    idx0, _, _ = g.retrieve(q, cu, s.k, s.T)
    out0 = g.question(q, cu, s.k, s.T)
    g.check_status()
    g.test_set_wait_limit(20000)
    g.test_set_retrieve(mode)
    idx = torch.full_like(idx0, -7)
    for l in range(L):
        g.question_layer(l, q[l], cu, s.k, s.T, idx=idx[l])
    with pytest.raises(rekv.RekvError) as e:
        g.check_status()
    assert e.value.code == rekv.ERR_TIMEOUT
    idx_r, _, _ = g.retrieve(q, cu, s.k, s.T)
    g.question(q, cu, s.k, s.T)
    with pytest.raises(rekv.RekvError) as e:
        g.check_status()
    assert e.value.code == rekv.ERR_TIMEOUT
    g.check_status()
    assert (idx_r[0, 0] == -1).all() and torch.equal(idx_r[1:], idx0[1:])
    assert (idx[:, 0] == -1).all()
    g.test_set_wait_limit(0)
    g.test_set_retrieve(0)
    assert torch.equal(g.retrieve(q, cu, s.k, s.T)[0], idx0)
    assert torch.equal(g.question(q, cu, s.k, s.T), out0)
    g.check_status()
    g.close()
