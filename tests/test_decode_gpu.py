"""Decode-shaped questions (at most 16 query rows per KV head) take the load-bound attention kernel: the same
parity checks as the other shapes, on the shapes that reach its branches."""
import pytest
import torch

from oracle import rekv_oracle as orc
from paper_2503_00540_b200 import rekv
from tests import harness as H
from tests.test_parity_gpu import _run_question_parity

pytestmark = pytest.mark.gpu


def test_one_token_question_7b_shape():
    """7 rows per KV head, 196-token frames, ranges cut by CTA boundaries (partials merged)."""
    _run_question_parity(H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=40, W=8, k=12), [1])


def test_two_tokens_and_batches_of_decode_steps():
    _run_question_parity(H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=30, W=4, k=6, seed=540), [2])
    _run_question_parity(H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=30, W=4, k=6, seed=7), [1, 2, 1])


def test_72b_head_shape_sixteen_rows():
    _run_question_parity(H.Shape(L=1, Hq=64, Hkv=8, Nf=196, T=20, W=4, k=6, seed=7), [2])


def test_short_and_odd_frames():
    """16-token frames (one warp has all the tokens), 100-token frames (ragged last unit), 208-token frames
    (the largest the library takes)."""
    _run_question_parity(H.TINY, [1])
    _run_question_parity(H.Shape(L=2, Hq=8, Hkv=2, Nf=100, T=20, W=3, k=5, seed=540), [2])
    _run_question_parity(H.Shape(L=1, Hq=8, Hkv=2, Nf=208, T=12, W=2, k=4, seed=7), [1])
    _run_question_parity(H.Shape(L=1, Hq=8, Hkv=2, Nf=208, T=12, W=2, k=4, seed=7), [30])  # and the tcgen05 kernel


def test_many_units_are_produced_whole():
    """More units than four times the SM count: every unit is one CTA's, no partials."""
    _run_question_parity(H.Shape(L=20, Hq=16, Hkv=8, Nf=32, T=10, W=2, k=4), [1] * 4, max_questions=4)


def test_host_tier_and_a_question_in_the_past():
    _run_question_parity(H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=40, W=4, k=8, tail=8), [1, 1])
    _run_question_parity(H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=40, W=8, k=12), [1], n_visible=21)


@pytest.mark.parametrize("theta,static", [(0.0, False), (1e6, False), (1e6, True)], ids=["no_rope", "rope", "static"])
@pytest.mark.parametrize("Nf,T,k,ns,heads", [
    (16, 30, 11, [5], (8, 2)),          # eight frames per step, the last step with fewer; X in a CTA of its own
    (33, 40, 20, [130], (28, 4)),       # frames with gap rows, two per step; X longer than a step
    (50, 12, 6, [1, 60], (16, 8)),      # 16 units on 9 CTAs each; X of two lengths
    (196, 80, 70, [48], (28, 4)),       # two frames on each CTA, rotated before the dependency wait
    (208, 60, 56, [9, 3], (32, 4)),     # three frames on a CTA and X behind them; three stages' worth of phases
    (24, 300, 290, [17], (4, 1)),       # one unit on 74 CTAs: parts of more than one batch
])
def test_tokens_layer_by_layer_over_one_context(theta, static, Nf, T, k, ns, heads):
    """One token per question through the layers, twice: the first launch after the gather waits before it asks for pages,
    the others have their frames copied (and rotated) before the wait.  Same bits, and the oracle's values."""
    s = H.Shape(L=3, Hq=heads[0], Hkv=heads[1], Nf=Nf, T=T, W=2, k=k, seed=7)
    nQ = len(ns)
    g = H.build_gpu(s, max_questions=nQ, max_q_tokens=nQ, max_self_tokens=sum(ns), rope_theta=theta,
                    flags=rekv.FLAG_ROPE_STATIC if static else 0)
    o = H.build_oracle(s)
    q, cu = H.questions(s, [1] * nQ, device="cuda")
    ks, vs, cus = H.self_kv(s, ns, device="cuda")
    refs = [o.question(q[:, i:i + 1].cpu().contiguous(), s.k, s.T) for i in range(nQ)]
    g.gather(torch.stack([r["idx"] for r in refs], dim=1).contiguous().cuda(), nQ, s.k, s.T)
    out = [torch.empty_like(q) for _ in range(2)]
    for o_pass in out:
        for l in range(s.L):
            g.attend_full_layer(l, q[l], ks[l], vs[l], cu, cus, out=o_pass[l])
    g.check_status()
    assert torch.equal(out[0], out[1])
    for i in range(nQ):
        for l in range(s.L):
            ref, _ = orc.attend_full(q[l, i:i + 1].cpu().contiguous(), refs[i]["k_ctx"][l].contiguous(),
                                     refs[i]["v_ctx"][l].contiguous(), ks[l, cus[i]:cus[i + 1]].cpu().contiguous(),
                                     vs[l, cus[i]:cus[i + 1]].cpu().contiguous(), theta, static_ctx=static)
            H.assert_attention(out[0][l:l + 1, i:i + 1], ref[None], f"layer {l} question {i}")
    g.close()
