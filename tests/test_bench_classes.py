"""The kernel classes that bench.py reports for a verify step, from the launch counts of a step."""
import numpy as np
import pytest

import bench
from paper_2203_16487_b200 import workloads as W


def test_classes_of_the_two_reported_steps():
    d, f, V, L = 512, 2048, 32768, 6
    # batch 1: the queries of the cross-attention and both output projections run inside the attention; only the final LayerNorm is a launch
    c = bench.step_classes(W.BASE_V, 25, 64, 64, 1, 34, {1: 12, 2: 1, 4: 12, 8: 1})
    assert [n for _, _, n, _ in c] == [12, 1, 12, 1, 8] and sum(n for _, _, n, _ in c) == 34
    assert c[0][3] == L * (64 + 26 + 64) * 2 * d * 2 + (6 + 12) * d * d * 2
    assert c[2][3] == L * (3 * d * d + f * d) * 2
    assert "6 query and 12 output" in c[0][1] and "cross-Q" not in c[2][1] and "attention out" not in c[4][1]
    # ... the queries and the cross-attention's output projections; the final LayerNorm inside the vocabulary projection
    c = bench.step_classes(W.BASE_V, 25, 64, 64, 1, 39, {1: 12, 2: 0, 4: 12, 8: 1})
    assert [n for _, _, n, _ in c] == [12, 0, 12, 1, 14] and sum(n for _, _, n, _ in c) == 39
    assert c[0][3] == L * (64 + 26 + 64) * 2 * d * 2 + (6 + 6) * d * d * 2
    assert "6 query and 6 output" in c[0][1] and "cross-Q" not in c[2][1] and "attention out" in c[4][1]
    # batch 128: every projection is a GEMM of its own
    c = bench.step_classes(W.BASE_V, 25, 64, 64, 128, 70, {1: 12, 2: 19, 4: 18, 8: 1})
    assert [n for _, _, n, _ in c] == [12, 19, 18, 1, 20] and sum(n for _, _, n, _ in c) == 70
    assert c[0][3] == 128 * L * (64 + 26 + 64) * 2 * d * 2
    assert c[2][3] == L * (4 * d * d + f * d) * 2
    assert "inside" not in c[0][1] and "cross-Q" in c[2][1] and "attention out" in c[4][1]
    # weights of the layers and the vocabulary are in exactly one class each
    whole = sum(b or 0 for _, _, _, b in c[:4]) + L * (2 * d * d + f * d) * 2 - c[0][3] - 128 * 26 * d * 2
    assert whole == (L * (6 * d * d + 2 * f * d) + V * d) * 2


def test_a_captured_figure_is_reported_for_the_captured_step_only():
    for B, c in bench.NCU_TRAFFIC.items():
        assert bench.ncu_traffic(B, c["launches"], "step") == c["step"] > 0
        assert bench.ncu_traffic(B, c["launches"] + 1, "step") is None
    assert bench.ncu_traffic(7, 34, "step") is None


@pytest.mark.gpu
@pytest.mark.parametrize("B", sorted(bench.NCU_TRAFFIC))
def test_the_captured_step_is_the_one_that_runs(B):
    from paper_2203_16487_b200 import binding
    sd = binding.SpecDec(W.BASE_V, W.make_weights(W.BASE_V, 1, True), W.BASE_D, W.make_weights(W.BASE_D, 2, True), k_max=25, max_batch=B, max_src=64, max_tgt=92, bf16=True)
    sd.encode(np.full((B, 64), 7, np.int32), [64] * B)
    before = sd.launch_count()
    sd.verify(np.full((B, 25), 7, np.int32), 3, 1.0)
    assert sd.launch_count() - before == bench.NCU_TRAFFIC[B]["launches"]
    sd.close()
