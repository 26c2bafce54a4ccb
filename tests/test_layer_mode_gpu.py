"""Layer-sequential entry points (one layer per call, as a decoder drives the path) against the all-layer
calls and the CPU oracle, eagerly and replayed from CUDA graphs."""
import pytest
import torch

from paper_2503_00540_b200 import rekv
from tests import harness as H

pytestmark = pytest.mark.gpu


def _layerwise(g, s, q, cu, n_visible, want_idx=True):
    nQ = len(cu) - 1
    out = torch.empty_like(q)
    idx = torch.full((s.L, nQ, s.k), -7, dtype=torch.int32, device="cuda")
    for l in range(s.L):
        g.question_layer(l, q[l], cu, s.k, n_visible, out=out[l], idx=idx[l] if want_idx else None)
    g.check_status()
    return out, idx


def _close(a, b, what):
    d = (a.float() - b.float()).abs()
    assert d.max().item() <= 4e-3 and d.mean().item() <= 2e-4, f"{what}: max {d.max().item()} mean {d.mean().item()}"


@pytest.mark.parametrize("shape,lengths", [
    (H.TINY, [16]),
    (H.Shape(L=3, Hq=28, Hkv=4, Nf=196, T=40, W=8, k=12), [32]),
    (H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=30, W=4, k=6, seed=540), [24, 64, 37, 5]),
    (H.Shape(L=2, Hq=64, Hkv=8, Nf=196, T=24, W=8, k=8, seed=7), [64]),
])
def test_layer_calls_match_all_layer_calls_and_oracle(shape, lengths):
    s = shape
    nQ = len(lengths)
    g = H.build_gpu(s, max_questions=nQ, max_q_tokens=sum(lengths))
    o = H.build_oracle(s)
    q, cu = H.questions(s, lengths, device="cuda")
    idx_all, k_eff, _ = g.retrieve(q, cu, s.k, s.T)
    out_all = g.question(q, cu, s.k, s.T, idx=idx_all)
    out_l, idx_l = _layerwise(g, s, q, cu, s.T)
    assert torch.equal(idx_l, idx_all)
    _close(out_l, out_all, "layer calls vs all-layer calls")
    # against the oracle wherever the selection is the oracle's
    q_cpu = q.cpu()
    for i in range(nQ):
        ref = o.question(q_cpu[:, cu[i]:cu[i + 1]].contiguous(), s.k, s.T)
        for l in range(s.L):
            if torch.equal(idx_l[l, i].cpu(), ref["idx"][l]):
                H.assert_attention(out_l[l:l + 1, cu[i]:cu[i + 1]], ref["out"][l:l + 1], f"layer {l} question {i}")
    # the internal selection buffer gives the same result as a caller's
    out_l2, _ = _layerwise(g, s, q, cu, s.T, want_idx=False)
    assert torch.equal(out_l2, out_l)
    g.close()


def test_layer_calls_replayed_from_cuda_graphs():
    """One graph per layer, captured once and replayed: same bits as the eager calls; a replay after the
    query buffer changed answers the new question."""
    s = H.Shape(L=3, Hq=28, Hkv=4, Nf=196, T=40, W=8, k=12)
    g = H.build_gpu(s, max_questions=1, max_q_tokens=32)
    q, cu = H.questions(s, [32], device="cuda")
    q2, _ = H.questions(s, [32], device="cuda", first_id=5)
    eager, idx_eager = _layerwise(g, s, q, cu, s.T)
    eager2, _ = _layerwise(g, s, q2, cu, s.T)
    qbuf = q.clone()
    out = torch.zeros_like(q)
    idx = torch.zeros((s.L, 1, s.k), dtype=torch.int32, device="cuda")
    graphs = []
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for l in range(s.L):
            gr = torch.cuda.CUDAGraph()
            with torch.cuda.graph(gr, stream=side):
                g.question_layer(l, qbuf[l], cu, s.k, s.T, out=out[l], idx=idx[l])
            graphs.append(gr)
    torch.cuda.current_stream().wait_stream(side)
    out.zero_()
    for gr in graphs:
        gr.replay()
    torch.cuda.synchronize()
    g.check_status()
    assert torch.equal(idx, idx_eager)
    assert torch.equal(out, eager)
    qbuf.copy_(q2)
    for gr in graphs:
        gr.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, eager2)
    g.close()


def test_decode_steps_reuse_the_layer_context():
    """After a question, single-token queries attend over the same retrieved context, layer by layer."""
    s = H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=40, W=8, k=12, seed=540)
    g = H.build_gpu(s, max_questions=1, max_q_tokens=32)
    o = H.build_oracle(s)
    q, cu = H.questions(s, [32], device="cuda")
    _, idx = _layerwise(g, s, q, cu, s.T)
    qd, cud = H.questions(s, [1], device="cuda", first_id=9)
    outd = torch.empty_like(qd)
    for l in range(s.L):
        g.attend_layer(l, qd[l], cud, out=outd[l])
    g.check_status()
    # the oracle attends the decode query over the context of the GPU's (checked) selection
    ref = o.question(q.cpu(), s.k, s.T)
    if torch.equal(idx[:, 0].cpu(), ref["idx"]):
        refd, _ = o.attend(qd.cpu(), ref["k_ctx"], ref["v_ctx"])
        H.assert_attention(outd, refd, "decode step")
    # and it equals the all-layer attend over the same context
    g.gather(idx, 1, s.k, s.T)
    _close(outd, g.attend(qd, cud), "attend_layer vs attend")
    g.close()


def test_layer_calls_on_the_host_tier():
    s = H.Shape(L=2, Hq=28, Hkv=4, Nf=196, T=40, W=4, k=8, tail=8)
    g = H.build_gpu(s, max_questions=2, max_q_tokens=48)
    q, cu = H.questions(s, [16, 32], device="cuda")
    idx_all, _, _ = g.retrieve(q, cu, s.k, s.T)
    out_all = g.question(q, cu, s.k, s.T, idx=idx_all)
    out_l, idx_l = _layerwise(g, s, q, cu, s.T)
    assert torch.equal(idx_l, idx_all)
    _close(out_l, out_all, "host tier, layer calls vs all-layer calls")
    g.close()


def test_layer_call_argument_errors():
    s = H.TINY
    g = H.build_gpu(s, max_questions=1, max_q_tokens=16)
    q, cu = H.questions(s, [16], device="cuda")
    with pytest.raises(rekv.RekvError):
        g.question_layer(s.L, q[0], cu, s.k, s.T)
    with pytest.raises(rekv.RekvError):
        g.question_layer(0, q[0], cu, s.k, s.T + 1)
    g2 = H.build_gpu(s, max_questions=1, max_q_tokens=16)
    with pytest.raises(rekv.RekvError):
        g2.attend_layer(0, q[0], cu)  # nothing gathered yet
    g.close()
    g2.close()


def test_all_layer_question_replayed_from_one_cuda_graph():
    """retrieve -> gather -> attend for all layers captured once (HBM-resident cache) and replayed after the query
    buffer changed: same bits as the eager calls."""
    s = H.Shape(L=3, Hq=28, Hkv=4, Nf=196, T=40, W=8, k=12)
    g = H.build_gpu(s, max_questions=2, max_q_tokens=48)
    q, cu = H.questions(s, [16, 32], device="cuda")
    q2, _ = H.questions(s, [16, 32], device="cuda", first_id=11)
    eager = g.question(q, cu, s.k, s.T).clone()
    eager2 = g.question(q2, cu, s.k, s.T).clone()
    qbuf, out = q.clone(), torch.zeros_like(q)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        gr = torch.cuda.CUDAGraph()
        with torch.cuda.graph(gr, stream=side):
            g.question(qbuf, cu, s.k, s.T, out=out)
    torch.cuda.current_stream().wait_stream(side)
    gr.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, eager)
    qbuf.copy_(q2)
    gr.replay()
    torch.cuda.synchronize()
    g.check_status()
    assert torch.equal(out, eager2)
    g.close()


def test_a_layer_context_built_under_another_geometry_is_refused():
    """All layers share one context table laid out by (questions, context frames).  A layer gathered with fewer
    visible frames (a shorter context) re-lays it out: the other layers' contexts are gone, and using them must fail
    with REKV_ERR_STATE instead of attending over the wrong pages; gathering the layer again makes it usable."""
    s = H.Shape(L=2, Hq=8, Hkv=2, Nf=16, T=20, W=4, k=8, seed=7)
    g = H.build_gpu(s, max_q_tokens=16)
    o = H.build_oracle(s)
    q, cu = H.questions(s, [16], device="cuda")
    ref = o.question(q.cpu(), s.k, s.T)
    out0 = g.question_layer(0, q[0], cu, s.k, s.T)
    g.question_layer(1, q[1], cu, s.k, 6)      # 2 candidates + 4 window frames: 6 context frames instead of 12
    g.check_status()
    with pytest.raises(rekv.RekvError) as e:
        g.attend_layer(0, q[0], cu)
    assert e.value.code == rekv.ERR_STATE
    with pytest.raises(rekv.RekvError) as e:
        g.attend(q, cu)
    assert e.value.code == rekv.ERR_STATE
    g.attend_layer(1, q[1], cu)                # the layer gathered last is fine
    out0b = g.question_layer(0, q[0], cu, s.k, s.T)
    g.check_status()
    assert torch.equal(out0, out0b)
    H.assert_attention(out0b[None], ref["out"][0:1], "layer 0 gathered again")
    g.close()


@pytest.mark.parametrize("k", [4, 12, 28])
@pytest.mark.parametrize("full", [False, True])
def test_a_token_directly_behind_the_question_of_its_layer(k, full):
    """question_layer and at once a one-token step over the context it builds, nothing between them, another question every
    time: contexts of one, two and four chunks, whose attention is one launch, so that the decode launch -- which asks for its
    first frames before its dependency wait -- follows it directly.  The same bits as with a synchronisation between the two,
    and those against the oracle."""
    s = H.Shape(L=3, Hq=8, Hkv=2, Nf=16, T=64, W=4, k=k, seed=540)
    extra = dict(max_self_tokens=8, rope_theta=1e6) if full else {}
    g = H.build_gpu(s, max_questions=1, max_q_tokens=16, **extra)
    o = H.build_oracle(s)
    n = 6
    qs = [H.questions(s, [16], device="cuda", first_id=10 * i)[0] for i in range(n)]
    toks = [H.questions(s, [1], device="cuda", first_id=10 * i + 5)[0] for i in range(n)]
    ks, vs, cus = H.self_kv(s, [8], device="cuda")

    def run(sync):
        out, outd = [torch.zeros_like(q) for q in qs], [torch.zeros_like(t) for t in toks]
        idx = torch.zeros((n, s.L, 1, k), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for i in range(n):
            for l in range(s.L):
                g.question_layer(l, qs[i][l], [0, 16], k, s.T, out=out[i][l], idx=idx[i, l])
                if sync:
                    torch.cuda.synchronize()
                if full:
                    g.attend_full_layer(l, toks[i][l], ks[l], vs[l], [0, 1], cus, out=outd[i][l])
                else:
                    g.attend_layer(l, toks[i][l], [0, 1], out=outd[i][l])
                if sync:
                    torch.cuda.synchronize()
        g.check_status()
        return out, outd, idx

    out0, outd0, idx0 = run(True)
    out1, outd1, idx1 = run(False)
    assert torch.equal(idx0, idx1)
    for i in range(n):
        assert torch.equal(out0[i], out1[i]) and torch.equal(outd0[i], outd1[i]), f"question {i}"
        ref = o.question(qs[i].cpu(), k, s.T)
        for l in range(s.L):
            if torch.equal(idx0[i, l, 0].cpu(), ref["idx"][l]):
                H.assert_attention(out0[i][l:l + 1], ref["out"][l:l + 1], f"question {i} layer {l}")
                if not full:
                    refd, _ = o.attend(toks[i].cpu(), ref["k_ctx"], ref["v_ctx"])
                    H.assert_attention(outd0[i][l:l + 1], refd[l:l + 1], f"token {i} layer {l}")
    g.close()
