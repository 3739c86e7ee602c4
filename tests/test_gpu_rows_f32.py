"""fp32 handles against the oracle, in lock step, at the edges of the few-rows GEMM and the attention kernel: row counts around a
16-row tile and the hand-over to the 64 x 64 tiles, reductions of one chunk, of the whole ring and beyond it, widths with and without
the LayerNorm inside, head sizes with and without the attention kernel, vocabularies that end inside a tile."""
import numpy as np
import pytest

from oracle import specdec_oracle as O
from paper_2203_16487_b200 import workloads as W
from tests import lockstep

pytestmark = pytest.mark.gpu


# (d, heads, ffn, vocab, batch, k)
@pytest.mark.parametrize("d,H,f,V,B,k", [
    (16, 4, 16, 65, 1, 15),         # 16 rows, 4-wide heads
    (48, 2, 528, 63, 1, 16),        # 17 rows, 24-wide heads (warp-per-row attention), five K chunks
    (128, 2, 384, 130, 3, 10),      # the ring exactly
    (144, 9, 400, 97, 2, 7),        # LayerNorm of more than 128 columns, K = 144
    (528, 33, 64, 70, 1, 3),        # too wide for the LayerNorm inside
    (64, 1, 128, 200, 96, 7),       # 768 verify rows
    (64, 4, 128, 200, 97, 7),       # 776: 64 x 64 tiles, K and V scattered by a kernel of their own
])
def test_fp32_edges(d, H, f, V, B, k):
    from paper_2203_16487_b200 import binding
    dims = W.ModelDims(d, H, f, V, 1, 2, 64)
    wv, wd = W.make_weights(dims, 50 + d, False), W.make_weights(dims, 51 + d, False)
    mv, md = O.model_from(dims, wv), O.model_from(dims, wd)
    rng = np.random.default_rng(B)
    srcs = [W.zipf_ids(rng, int(n), V) for n in rng.integers(1, 13, size=B)]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=12, max_tgt=16, bf16=False)
    sd.set_option("debug_checks", 1)
    rep = lockstep.run(sd, mv, md, srcs, [10] * B, k, 3, 1.0, margin=1e-5, check_logits_every=1, max_iters=2)
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 1e-4 and rep.max_stat_err < 1e-4
    tgt = [1 + b % 9 for b in range(B)]
    out, n, _ = sd.generate(*W.pad_batch(srcs), np.array(tgt, np.int32), k, 1, 0.0)
    out, n = out.cpu().numpy(), n.cpu().numpy()
    for b in range(0, B, 7):
        assert out[b, :n[b]].tolist() == O.greedy_decode(mv, srcs[b], tgt[b], W.BOS_ID, W.EOS_ID), b
    sd.close()
