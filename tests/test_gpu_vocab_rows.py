"""The vocabulary projection of few rows (final LayerNorm, drafts' logits and statistics in one kernel) against the oracle, in lock step: vocabularies at
both ends of its range and one whose last tile is ragged, row counts at the edges of its two sizes, the row beyond them, and the drafter's pass."""
import numpy as np
import pytest

from oracle import specdec_oracle as O
from paper_2203_16487_b200 import workloads as W
from tests import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,B,k", [
    (18945, 1, 15),         # the smallest vocabulary that takes it (one column in the last tile), 16 rows
    (33152, 1, 16),         # the largest (148 whole tiles), 17 rows
    (20001, 4, 7),          # 32 rows
    (20001, 3, 10),         # 33 rows: the launches that serve any count
    (32768, 1, 1),          # 2 rows, one of the drafter
])
def test_vocab_rows_edges(V, B, k):
    from paper_2203_16487_b200 import binding
    dims = W.ModelDims(512, 8, 128, V, 1, 1, 64)
    wv, wd = W.make_weights(dims, 61, True), W.make_weights(dims, 62, True)
    mv, md = O.model_from(dims, wv, mode="bf16"), O.model_from(dims, wd, mode="bf16")
    rng = np.random.default_rng(B)
    srcs = [W.zipf_ids(rng, int(n), V) for n in rng.integers(2, 13, size=B)]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=12, max_tgt=24, bf16=True)
    sd.set_option("debug_checks", 1)
    rep = lockstep.run(sd, mv, md, srcs, [20] * B, k, 3, 1.0, margin=1e-3, check_logits_every=1, max_iters=3)
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 2e-2 and rep.max_stat_err < 2e-2
    # packed blocks: budgets that end at different iterations, down to one sequence
    tgt = [2 + 5 * b for b in range(B)]
    out, n, _ = sd.generate(*W.pad_batch(srcs), np.array(tgt, np.int32), k, 1, 0.0)
    out, n = out.cpu().numpy(), n.cpu().numpy()
    for b in range(B):
        assert out[b, :n[b]].tolist() == O.greedy_decode(mv, srcs[b], tgt[b], W.BOS_ID, W.EOS_ID), b
    # a draft outside the vocabulary is refused, as ever: nothing is accepted before it
    sd.encode(*W.pad_batch(srcs), None)
    drafts = np.full((B, k), V, np.int32)
    acc, bif = sd.verify(drafts, V, 1e9)
    assert acc.cpu().tolist() == [0] * B
    sd.close()


def test_a_block_without_drafts_has_no_draft_logits():
    """verify with k = 0 (no drafts: a null pointer) behind a block that had some: every row reports (+inf, -1), not what the earlier block left."""
    from paper_2203_16487_b200 import binding
    V, B = 20001, 2
    dims = W.ModelDims(512, 8, 128, V, 1, 1, 64)
    sd = binding.SpecDec(dims, W.make_weights(dims, 61, True), dims, W.make_weights(dims, 62, True), k_max=4, max_batch=B, max_src=12, max_tgt=24, bf16=True)
    rng = np.random.default_rng(2)
    sd.encode(*W.pad_batch([W.zipf_ids(rng, 9, V) for _ in range(B)]), None)
    drafts = rng.integers(4, V, size=(B, 4)).astype(np.int32)
    sd.verify(drafts, 3, 1.0)
    assert sd.debug_row_stats(4)[:, :4, 5].cpu().numpy().astype(int).tolist() == drafts.tolist()
    sd.verify(np.zeros((B, 0), np.int32), 3, 1.0)
    stats = sd.debug_row_stats(0).cpu().numpy()
    assert np.isposinf(stats[:, 0, 4]).all() and (stats[:, 0, 5] == -1).all(), stats
    sd.close()


@pytest.mark.parametrize("lse", [0, 1])
def test_columns_that_are_nan_hide_no_others(lse):
    """28 columns of a tile, all that one warp sees, are NaN (broken weights): the rest of the tile counts as in the launches that serve any number of rows."""
    from paper_2203_16487_b200 import binding
    V, k = 20001, 3
    dims = W.ModelDims(512, 8, 128, V, 1, 1, 64)
    wv = W.make_weights(dims, 61, True)
    drafts = np.array([[224 * 40 + 100, 224 * 41 + 30, 224 * 42 + 200]], np.int32)     # (a row's largest logit is the token it was fed)
    for first in (224 * 40, 224 * 41, 224 * 41 + 56, 224 * 42 + 84):
        wv["embed"][first:first + 28] = np.nan
    rng = np.random.default_rng(3)
    src = W.zipf_ids(rng, 9, 5000)
    got = {}
    for skinny in (1, 0):
        sd = binding.SpecDec(dims, wv, dims, wv, k_max=k, max_batch=1, max_src=12, max_tgt=24, bf16=True)
        sd.set_option("skinny", skinny)
        sd.set_option("row_lse", lse)
        sd.encode(*W.pad_batch([src]), None)
        acc, bif = sd.verify(drafts, 3, 1.0)
        got[skinny] = sd.debug_row_stats(k).cpu().numpy()[0], acc.item(), bif.item()
        sd.close()
    assert got[1][0][:, 1].astype(int).tolist() == got[0][0][:, 1].astype(int).tolist() == [W.BOS_ID] + drafts[0].tolist()
    assert got[1][1:] == got[0][1:]
    assert np.abs(got[1][0][:, [0, 4]][:k] - got[0][0][:, [0, 4]][:k]).max() < 2e-2    # (bf16 operands: two orders of the same sums)
    assert (got[1][0][:, 3] == got[0][0][:, 3])[:k].all()
