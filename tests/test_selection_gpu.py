"""Step 3 at the sizes and score patterns where the selection kernel changes its way: up to 2048 candidates one histogram
over equal score steps and an exact ranking inside the step that holds the k-th largest; radix passes beyond that, when the
step has more than 64 members, and when a score is not finite.  The scores come back from the same call, so the selection has
to match exactly what sorting them gives (score, then lower index; NaN last; ascending output)."""
import pytest
import torch

from paper_2503_00540_b200 import rekv
from tests import harness as H

pytestmark = pytest.mark.gpu


def _select(embs: torch.Tensor, k: int, W: int = 0, b: int = 1):
    T = embs.shape[0]
    g = rekv.ReKV(3, 4, 1, 128, 1, T, W, max_topk=k, block_frames=b, ext_embed_dim=embs.shape[1])
    kv = torch.zeros((3, 1, 1, 128), dtype=torch.bfloat16, device="cuda")
    for f in range(T):
        g.append_frame(kv, kv)
        g.set_frame_embedding(f, embs[f])
    q = torch.zeros((1, embs.shape[1]), device="cuda")
    q[0, 0] = 1.0
    idx, k_eff, scores = g.retrieve_external(q, k, T, 1.0, want_scores=True)
    n_scored = scores.shape[1]
    g.check_status()
    g.close()
    n_cand = max(T - W, 0) if b == 1 else n_scored
    s = scores[0, :n_cand].cpu()
    s = torch.where(torch.isnan(s), torch.full_like(s, float("-inf")), s)
    items = sorted(range(n_cand), key=lambda i: (-s[i].item(), i))[:k_eff // b]
    want = [i * b + j for i in sorted(items) for j in range(b)]
    for l in range(3):
        assert idx[l, 0, :k_eff].tolist() == want, f"layer {l}"
        assert (idx[l, 0, k_eff:] == -1).all()


def _angles(n, seed):
    gen = torch.Generator().manual_seed(seed)
    a = torch.rand(n, generator=gen) * 3.0
    return torch.stack([a.cos(), a.sin(), 0 * a, 0 * a], 1).cuda().contiguous()


@pytest.mark.parametrize("T,k,W", [(1, 1, 0), (2, 1, 1), (65, 64, 0), (513, 8, 0), (2047, 64, 3), (2048, 64, 0),
                                   (2049, 64, 0), (2600, 200, 8), (1800, 1800, 8)])
def test_selection_at_the_edges_of_the_histogram_path(T, k, W):
    _select(_angles(T, T), k, W)


@pytest.mark.parametrize("pattern", ["all_equal", "pairs", "one_step", "nan", "zero_norm"])
def test_selection_with_ties_crowded_steps_and_scores_that_are_not_numbers(pattern):
    e = _angles(1500, 5)
    if pattern == "all_equal":
        e[:] = e[0]
    elif pattern == "pairs":      # every score twice, 40 of them thirty times
        e[1::2] = e[0::2]
        e[300:330] = e[700]
    elif pattern == "one_step":   # one far score; all others inside a single step
        a = 1.0 + 1e-6 * torch.arange(1500)
        e = torch.stack([a.cos(), a.sin(), 0 * a, 0 * a], 1).cuda().contiguous()
        e[77] = torch.tensor([-1.0, 0, 0, 0])
    elif pattern == "nan":
        e[3] = float("nan")
        e[900] = float("nan")
    else:
        e[10:50] = 0.0
    _select(e, 64)
    _select(e[:1496].contiguous(), 64, b=8)


@pytest.mark.parametrize("L,Hkv,T,b,lengths", [
    (1, 2, 256, 1, [3]), (1, 2, 1025, 1, [3]),        # 16 CTAs per layer, one row per warp at most; beyond four
    (7, 4, 1024, 1, [5, 1]), (9, 4, 1024, 1, [5, 1]), (10, 4, 256, 1, [5]),    # ... while one fits a GPC; then 8 CTAs per layer
    (28, 2, 64, 1, [5]), (40, 2, 64, 1, [5]),         # ... while all layers' clusters are resident at once
    (10, 4, 257, 1, [5]), (2, 8, 512, 1, [2, 7, 1, 4]), (12, 8, 128, 1, [2]), (12, 8, 129, 1, [2]),
    (2, 3, 40, 1, [6]), (2, 4, 515, 8, [6]),           # idle CTAs; blocks
    (1, 1, 7, 1, [1] * 5), (2, 4, 51, 1, [1] * 7), (1, 8, 33, 1, [2] * 11), (2, 2, 50, 1, [1] * 20)])  # eight at a time, and the rest
def test_one_launch_retrieval_and_the_sizes_around_it(L, Hkv, T, b, lengths):
    """Question vector, scores and selection in one launch (clusters) and just beyond the sizes it takes: the scores against
    64-bit sums over the same representatives to 1e-4 (two orders above what fp32 sums lose), the selection exactly what those
    scores give."""
    s = H.Shape(L=L, Hq=2 * Hkv, Hkv=Hkv, Nf=2, T=T, W=3, k=8, seed=7, b=b)
    g = H.build_gpu(s, max_questions=len(lengths), max_q_tokens=sum(lengths))
    q, cu = H.questions(s, lengths, device="cuda")
    idx, k_eff, scores = g.retrieve(q, cu, 8, T, want_scores=True)
    idx2, _, _ = g.retrieve(q, cu, 8, T)
    g.check_status()
    assert torch.equal(idx, idx2)
    n_cand = max(T - 3, 0) // b
    for l in range(L):
        reps = g.get_reps(l, T).double()
        if b > 1:
            reps = reps[:n_cand * b].reshape(n_cand, b, -1).mean(1)
        for i in range(len(lengths)):
            v = q[l, cu[i]:cu[i + 1]].double().reshape(-1, Hkv, 2, 128).mean((0, 2)).reshape(-1)
            ref = (reps @ v) / (reps.norm(dim=1).clamp_min(1e-8) * v.norm().clamp_min(1e-8))
            row = scores[l, i].cpu()
            H.assert_close_rel(row[None], ref.cpu()[None], f"scores of layer {l}, question {i}")
            items = sorted(sorted(range(n_cand), key=lambda f: (-row[f].item(), f))[:k_eff // b])
            assert idx[l, i, :k_eff].tolist() == [f * b + j for f in items for j in range(b)]
    g.close()


@pytest.mark.parametrize("L,Hkv,G,T,b,lengths", [
    (1, 2, 4, 64, 1, [16]), (12, 2, 4, 60, 1, [5, 9]),   # clusters of 16 and of 8 CTAs
    (1, 1, 8, 90, 1, [40]), (2, 3, 2, 77, 1, [33, 1]), (9, 4, 7, 200, 1, [32]), (2, 8, 8, 100, 1, [20, 3, 30, 7]),
    (10, 1, 4, 33, 1, [7]), (11, 5, 3, 50, 1, [50]), (12, 8, 2, 100, 1, [130]), (2, 4, 7, 163, 8, [20]), (10, 4, 7, 96, 2, [9]), (28, 4, 7, 64, 1, [32])])
def test_one_launch_and_three_launches_give_the_same_bits(L, Hkv, G, T, b, lengths):
    """A context where no cluster can be resident takes the three launches, as larger tables do: the same scores to the bit,
    and so the same selection; a layer at a time and rekv_score_frames_static as well.  (Question rows per KV group from 2 to
    320, one to eight CTAs summing them.)"""
    s = H.Shape(L=L, Hq=G * Hkv, Hkv=Hkv, Nf=2, T=T, W=3, k=8, seed=7, b=b)
    g = H.build_gpu(s, max_questions=len(lengths), max_q_tokens=sum(lengths))
    q, cu = H.questions(s, lengths, device="cuda")

    def retrieve():
        n = g.launch_count()
        idx, _, scores = g.retrieve(q, cu, 8, T, want_scores=True)
        n = g.launch_count() - n
        idx_l = torch.empty_like(idx)
        for l in range(L):
            g.question_layer(l, q[l], cu, 8, T, idx=idx_l[l])
        return idx, scores, idx_l, g.question(q, cu, 8, T), n

    idx1, scores1, idx_l1, out1, n1 = retrieve()
    g.test_set_retrieve(rekv.TEST_RETRIEVE_NO_CLUSTER)
    idx3, scores3, idx_l3, out3, n3 = retrieve()
    g.check_status()
    assert (n1, n3) == (1, 3)
    assert torch.equal(scores1, scores3) and torch.equal(idx1, idx3) and torch.equal(out1, out3)
    assert torch.equal(idx_l1, idx1) and torch.equal(idx_l3, idx1)
    if b == 1:
        for l in range(L):
            assert torch.equal(rekv.score_frames_static(q[l].contiguous(), cu, Hkv, g.get_reps(l, T)), scores1[l])
    g.close()
