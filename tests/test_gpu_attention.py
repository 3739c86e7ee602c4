"""The attention kernel against the oracle, in lock step: every variant (16 / 32 / 64 queries per CTA, one, four or eight key groups)
over key counts at the edges of its key blocks (32 a warp, 64, 128, 256 a block), with the ring wrapping and with less
than one block, query counts at the edges of the query tiles, cached prefixes that end inside a block."""
import numpy as np
import pytest

from oracle import specdec_oracle as O
from paper_2203_16487_b200 import workloads as W
from tests import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{}, {"attn_warps": 4}, {"attn_warps": 8}, {"attn_stream": 2}, {"attn_stream": 3}, {"attn_stream": 4}])
@pytest.mark.parametrize("lens,k", [((1, 31, 33, 64, 65), 15), ((127, 129, 255, 257, 385), 33)])
def test_attention_edges(opts, lens, k):
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(128, 2, 128, V, 1, 2, 512)
    wv, wd = W.make_weights(dims, 71, True), W.make_weights(dims, 72, True)
    mv, md = O.model_from(dims, wv, mode="bf16"), O.model_from(dims, wd, mode="bf16")
    rng = np.random.default_rng(k)
    srcs = [W.zipf_ids(rng, n, V) for n in lens]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=len(lens), max_src=max(lens), max_tgt=100, bf16=True)
    for name, v in opts.items():
        sd.set_option(name, v)
    sd.set_option("debug_checks", 1)
    # drafts that are accepted in part: the prefixes grow by different lengths
    greedy = [O.greedy_decode(mv, s, 100, W.BOS_ID, W.EOS_ID) for s in srcs]

    def drafts(b, out, n):
        d = (greedy[b] + [5] * n)[len(out):len(out) + n]
        cut = (7 * b + 3 + len(out)) % n
        return np.array(d[:cut] + [(d[cut] + 9) % V] + d[cut + 1:], np.int32)

    rep = lockstep.run(sd, mv, md, srcs, [100] * len(lens), k, 1, 0.0, margin=1e-3, check_logits_every=1, max_iters=4, draft_fn=drafts)
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 2e-2 and rep.max_stat_err < 2e-2
    # the drafter's own attention (bidirectional, all rows of the sequence)
    g = sd.draft(k).cpu().numpy()
    out, n, fin = sd.output()
    out, n, fin = out.cpu().numpy(), n.cpu().numpy(), fin.cpu().numpy()
    for b in (0, 2, 4):
        if fin[b]:
            continue
        logits = O.decoder_rows(md, [W.BOS_ID] + out[b, :n[b]].tolist() + [W.MASK_ID] * k, O.encode(md, srcs[b]), causal=False)[n[b] + 1:]
        for i in range(k):
            assert g[b, i] == logits[i].argmax() or logits[i].max() - logits[i, g[b, i]] < 2e-2, (b, i)
    sd.close()


@pytest.mark.parametrize("d,f,B,k,S", [(256, 256, 1, 15, 12), (512, 128, 3, 16, 130), (256, 128, 2, 15, 300), (768, 128, 2, 31, 400)])
def test_queries_projected_inside_the_attention(d, f, B, k, S):
    """Cross-attention of few rows: one and two 16-row tiles with a ragged end, key rings of one stage and more, the three widths."""
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(d, d // 64, f, V, 1, 1, 512)
    wv, wd = W.make_weights(dims, 81, True), W.make_weights(dims, 82, True)
    mv, md = O.model_from(dims, wv, mode="bf16"), O.model_from(dims, wd, mode="bf16")
    rng = np.random.default_rng(d)
    srcs = [W.zipf_ids(rng, n, V) for n in ([S] + [max(S // 2, 1), 7])[:B]]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=S, max_tgt=40, bf16=True)
    sd.set_option("debug_checks", 1)
    rep = lockstep.run(sd, mv, md, srcs, [40] * B, k, 3, 1.0, margin=1e-3, check_logits_every=1, max_iters=2)
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 2e-2 and rep.max_stat_err < 2e-2
    sd.close()


@pytest.mark.parametrize("S,k", [(128, 4), (129, 4), (128, 3), (5, 5), (4, 2), (33, 20)])
def test_key_groups_share_their_probabilities(S, k):
    """Encoder self-attention and cross-attention of four key groups over one block of keys and over one key more, with as few queries as share and one less; groups without keys."""
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(128, 2, 128, V, 2, 1, 512)
    wv, wd = W.make_weights(dims, 85, True), W.make_weights(dims, 86, True)
    mv, md = O.model_from(dims, wv, mode="bf16"), O.model_from(dims, wd, mode="bf16")
    rng = np.random.default_rng(S + k)
    srcs = [W.zipf_ids(rng, n, V) for n in (S, max(S // 3, 1), 1)]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=3, max_src=S, max_tgt=40, bf16=True)
    sd.set_option("debug_checks", 1)
    rep = lockstep.run(sd, mv, md, srcs, [40] * 3, k, 3, 1.0, margin=1e-3, check_logits_every=1, max_iters=3)
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 2e-2 and rep.max_stat_err < 2e-2
    sd.close()


@pytest.mark.parametrize("d,B,k,S,cached", [
    (256, 1, 4, 12, False),          # 5 rows of one tile: the fewest
    (512, 1, 15, 128, False),        # 16 rows of eight heads, 8 CTAs: both attentions go on to their output projections; as many keys as fit beside the queries'
    (512, 1, 15, 129, True),         # one key too many for that: the cross-attention projects its queries only
    (512, 1, 16, 128, False),        # 17 rows, 16 CTAs: the cross-attention only, and the last
    (512, 1, 32, 128, False),        # 33 rows, 24 CTAs: neither
    (256, 2, 23, 128, False),        # four heads, 48 rows: the most with the queries projected too
    (256, 1, 48, 128, True),         # 49 rows: the self-attention only
    (256, 3, 16, 300, True),         # three stages of keys
])
def test_output_projected_inside_the_attention(d, B, k, S, cached):
    """Attention of few rows that goes on to the output projection and the residual, self- and cross-attention, the drafter's [MASK] rows among them."""
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(d, d // 64, 128, V, 1, 2, 512)
    wv, wd = W.make_weights(dims, 83, True), W.make_weights(dims, 84, True)
    mv, md = O.model_from(dims, wv, mode="bf16"), O.model_from(dims, wd, mode="bf16")
    rng = np.random.default_rng(d + S)
    srcs = [W.zipf_ids(rng, n, V) for n in ([S] + [max(S // 2, 1), 7])[:B]]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=S, max_tgt=60, bf16=True)
    sd.set_option("debug_checks", 1)
    rep = lockstep.run(sd, mv, md, srcs, [60] * B, k, 3, 1.0, margin=1e-3, check_logits_every=1, max_iters=2,
                       drafter_reading="prefix_causal" if cached else "bidirectional")
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 2e-2 and rep.max_stat_err < 2e-2
    sd.close()


@pytest.mark.parametrize("bf16,d,H,cached", [(True, 256, 4, False), (True, 256, 4, True), (True, 512, 8, False), (True, 512, 8, True),
                                             (False, 64, 16, False), (False, 64, 16, True)])
def test_slices_of_unfinished_sequences(bf16, d, H, cached):
    """A ragged batch whose sequences end one after another: the attention launches shrink to the unfinished ones (32, 16, ... of 33).
    Every draft is accepted, so what comes out is what the drafter's passes computed, and each (k + 1)-th token what the verifier's did."""
    from paper_2203_16487_b200 import binding
    V, B, k, beta, tau = 515, 33, 17, 515, 1e9
    dims = W.ModelDims(d, H, 2 * d, V, 1, 2, 128)
    wv, wd = W.make_weights(dims, 91, bf16), W.make_weights(dims, 92, bf16)
    for w in (wv, wd):                                   # sublayers that outweigh the embedding: the argmax depends on every key
        for name in w:
            if name.endswith((".o.w", ".v.w", ".ffn.w2")):
                w[name] = w[name] * 8
        w["pos_dec"] = 4 * np.random.default_rng(5).standard_normal(w["pos_dec"].shape).astype(np.float32)
    mv, md = (O.model_from(dims, w, mode="bf16" if bf16 else "pure") for w in (wv, wd))
    rng = np.random.default_rng(4)
    srcs = [W.zipf_ids(rng, int(n), V) for n in rng.integers(2, 20, size=B)]
    tgt = [3 + 9 * (b % 9) for b in range(B)]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=20, max_tgt=max(tgt), bf16=bf16)
    sd.set_option("debug_checks", 1)
    sd.set_option("drafter_prefix_causal", int(cached))
    out, n, _ = sd.generate(*W.pad_batch(srcs), np.array(tgt, np.int32), k, beta, tau)
    out, n = out.cpu().numpy(), n.cpu().numpy()

    def gap_at_the_first_difference(b, got, ref):
        """By how much the oracle's logits of that position prefer its token to the other one, on the prefix that both share."""
        p = next((i for i, (x, y) in enumerate(zip(got, ref)) if x != y), None)
        assert p is not None, (b, got, ref)              # (one ends early: no margin explains that)
        j = p // (k + 1) * (k + 1)                       # tokens committed before this block
        if p - j < k:
            row = O.decoder_rows(md, [W.BOS_ID] + ref[:j] + [W.MASK_ID] * k, O.encode(md, srcs[b]), causal=False, n_causal=j + 1 if cached else None)[j + 1 + p - j]
        else:
            row = O.decoder_rows(mv, [W.BOS_ID] + ref[:p], O.encode(mv, srcs[b]), causal=True)[-1]
        assert row.argmax() == ref[p]
        return row[ref[p]] - row[got[p]]

    gaps, seen = [], set()
    for b in range(B):
        ref, _ = O.specdec_generate(mv, md, srcs[b], tgt[b], k, beta, tau, W.BOS_ID, W.EOS_ID, W.MASK_ID,
                                    drafter_reading="prefix_causal" if cached else "bidirectional")
        got = out[b, :n[b]].tolist()
        if got != ref:
            gaps.append(gap_at_the_first_difference(b, got, ref))
        seen.update(ref)
    assert len(seen) > 40                                # (the drafts do vary)
    # fp32: exact.  bf16: two logits that each agree with the oracle's to 2e-3 may change places where these are less than twice that apart (about 1300 arguments of
    # a maximum over 515 logits of spread ~1: a few near-ties are expected).  A slice that is lost or swapped differs by the spread.
    assert not gaps if not bf16 else all(g < 4e-3 for g in gaps), gaps
    sd.close()
