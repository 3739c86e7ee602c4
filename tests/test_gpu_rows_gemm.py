"""The few-rows GEMM against the oracle, in lock step, at the row counts where its launch rule changes (16-row tiles, LayerNorm inside
or in front, the hand-over to the 128-row tensor-core tiles) and at widths that are not whole MMA steps of its K slices,
have no LayerNorm inside, or split long reductions across a cluster (K = 1024 and more)."""
import numpy as np
import pytest

from oracle import specdec_oracle as O
from paper_2203_16487_b200 import workloads as W
from tests import lockstep

pytestmark = pytest.mark.gpu


# (d, heads, ffn, batch, k): batch * (k + 1) rows in a verify block
@pytest.mark.parametrize("d,H,f,B,k", [
    (256, 4, 1040, 1, 15),          # 16 rows; K = 1040: two slices that end inside an MMA step
    (512, 8, 2048, 1, 15),          # 16 rows: the last with weight fragments of 32 columns
    (512, 8, 2048, 1, 16),          # 17 rows: a tile and one row, fragments of 64 columns; K = 2048 in four slices
    (512, 8, 2048, 3, 10),          # 33 rows
    (512, 8, 2048, 3, 15),          # 48 rows: the last with fragments where a LayerNorm runs inside
    (512, 8, 2048, 7, 6),           # 49 rows
    (256, 4, 1024, 1, 4),           # 5 rows; K = 1024: two slices, as fragments
    (256, 4, 1024, 8, 3),           # 32 rows: the last with 16-column output projections
    (768, 12, 3072, 1, 15),         # 16 rows at this width: fragments of the widest LayerNorm
    (768, 12, 3072, 1, 16),         # 17 rows: without
    (768, 12, 3072, 8, 9),          # 80 rows: the last with the LayerNorm inside
    (768, 12, 3072, 16, 5),         # 96 rows: the last of the few-rows kernel at this width
    (768, 12, 3072, 16, 7),         # 128 rows: tensor-core tiles, four K slices for the output projections
    (512, 8, 2048, 16, 8),          # 144 rows: the last with the LayerNorm inside at this width
    (256, 4, 1024, 29, 4),          # 145 rows: LayerNorm in front, four slices
    (320, 5, 1312, 16, 10),         # 176 rows: the last of the few-rows kernel; no LayerNorm width, an FFN that has no tiles
    (320, 5, 1312, 24, 15),         # 384 rows: the FFN's output projection stays with the few-rows kernel
    (128, 2, 192, 35, 10),          # 385 rows: tensor-core tiles
    (512, 8, 2048, 8, 11),          # 96 rows: the last output projections on 16 x 32 tiles
    (512, 8, 2048, 7, 13),          # 98 rows: 16 x 64 tiles, the last of them two rows
    (512, 8, 2048, 8, 15),          # 128 rows: the last with the FFN2 here
    (512, 8, 2048, 10, 12),         # 130 rows: its split-K tiles
    (512, 8, 2112, 10, 12),         # 130 rows: a reduction that has no split-K tiles stays, two slices of 66 MMA steps
    (512, 8, 2112, 11, 15),         # 176 rows: the last of them, four slices
    (512, 8, 2048, 14, 15),         # 224 rows: the last QKV projections on 32-row tiles
    (512, 8, 2048, 14, 16),         # 238 rows: QKV on tensor-core tiles again, output projections on 16-row tiles, the last of them 14 rows
    (512, 8, 2048, 27, 15),         # 432 rows: the last output projections on 16-row tiles
    (512, 8, 2048, 31, 13),         # 434 rows: ... on 32-row tiles
    (512, 8, 2048, 46, 15),         # 736 rows: the last on 32-row tiles
    (768, 12, 3072, 3, 26),         # 81 rows: 16 x 32 tiles at this width, beyond the LayerNorm inside
    (768, 12, 3072, 10, 15),        # 160 rows: the last of them
    (768, 12, 3072, 7, 22),         # 161 rows: 32 x 64 tiles
    (768, 12, 3072, 20, 15),        # 320 rows: the last of them
    (512, 8, 2048, 16, 11),         # 192 rows: four slices of three whole 64-row tiles
    (512, 8, 2048, 16, 15),         # 256 rows: the last of them
    (768, 12, 3072, 13, 9),         # 130 rows: 128-row tiles again at this width, the last of two rows
    (512, 8, 2048, 32, 15),         # 512 rows: the last four K slices of a tile at this width, the last row tile full
    (512, 8, 2048, 27, 18),         # 513 rows: two K slices, one row in the last tile
    (512, 8, 2048, 61, 18),         # 1159 rows: two K slices of 128-column tiles, seven rows in the last of them
    (512, 8, 2048, 96, 23),         # 2304 rows: the last of them, every tile full
    (512, 8, 1664, 48, 25),         # 1248 rows: a reduction too short for them
    (768, 12, 3072, 40, 21),        # 880 rows: at this width
    (256, 4, 1152, 20, 14),         # 300 rows: two slices of nine K blocks, more than the ring holds
])
def test_rows_gemm_edges(d, H, f, B, k):
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(d, H, f, V, 1, 1, 64)
    wv, wd = W.make_weights(dims, 40 + d, True), W.make_weights(dims, 41 + d, True)
    mv, md = O.model_from(dims, wv, mode="bf16"), O.model_from(dims, wd, mode="bf16")
    rng = np.random.default_rng(B)
    srcs = [W.zipf_ids(rng, int(n), V) for n in rng.integers(2, 13, size=B)]
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=12, max_tgt=16, bf16=True)
    sd.set_option("debug_checks", 1)
    rep = lockstep.run(sd, mv, md, srcs, [10] * B, k, 3, 1.0, margin=1e-3, check_logits_every=1, max_iters=2)
    assert rep.ok, rep.notes
    assert rep.max_logit_err < 2e-2 and rep.max_stat_err < 2e-2
    # packed blocks: budgets that end at different iterations
    tgt = [1 + b % 9 for b in range(B)]
    out, n, _ = sd.generate(*W.pad_batch(srcs), np.array(tgt, np.int32), k, 1, 0.0)
    out, n = out.cpu().numpy(), n.cpu().numpy()
    for b in range(0, B, 7):
        assert out[b, :n[b]].tolist() == O.greedy_decode(mv, srcs[b], tgt[b], W.BOS_ID, W.EOS_ID), b
    sd.close()
