"""specdec_launch_count against the kernel nodes of a captured graph: every launch is counted, and nothing else."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2203_16487_b200 import workloads as W

pytestmark = pytest.mark.gpu

CU_GRAPH_NODE_TYPE_KERNEL = 0


def _kernel_nodes(graph) -> int:
    cu, g, n = C.CDLL("libcuda.so.1"), C.c_void_p(graph.raw_cuda_graph()), C.c_size_t()
    assert cu.cuGraphGetNodes(g, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, C.byref(n)) == 0
    kinds = []
    for node in nodes:
        t = C.c_int()
        assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(t)) == 0
        kinds.append(t.value)
    return kinds.count(CU_GRAPH_NODE_TYPE_KERNEL)


# one CTA per 16 queries with the projections inside (the [MASK] rows gathered there), separate launches, the cached drafter, the fp32 path
@pytest.mark.parametrize("d,f,B,k,bf16,cached", [(256, 512, 1, 8, True, False), (256, 512, 1, 3, True, False), (512, 1024, 24, 10, True, False),
                                                 (256, 512, 2, 9, True, True), (64, 128, 2, 8, False, False)])
@pytest.mark.parametrize("repeat", [0, 1, 2, 4, 8])
def test_every_step_counts_the_kernels_it_launches(d, f, B, k, bf16, cached, repeat):
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(d, d // 64, f, V, 1, 2, 128)
    wv, wd = W.make_weights(dims, 5, bf16), W.make_weights(dims, 6, bf16)
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=20, max_tgt=40, bf16=bf16)
    sd.set_option("graphs", 0)                       # the step calls launch into the capture themselves
    sd.set_option("diag_repeat", repeat)
    if cached:
        sd.set_option("drafter_prefix_causal", 1)
    rng = np.random.default_rng(1)
    src = torch.from_numpy(np.stack([W.zipf_ids(rng, 20, V) for _ in range(B)])).cuda()
    i32 = dict(dtype=torch.int32, device="cuda")
    lens, draft, acc, bif = torch.full((B,), 20, **i32), torch.zeros((B, k), **i32), torch.zeros(B, **i32), torch.zeros(B, **i32)
    lib, ptr = sd._lib, binding._ptr
    steps = {
        "encode": lambda s: lib.specdec_encode(sd._h, ptr(src), ptr(lens), None, B, 20, s),
        "draft": lambda s: lib.specdec_draft(sd._h, k, ptr(draft), s),
        "verify": lambda s: lib.specdec_verify(sd._h, ptr(draft), k, 3, 1.0, ptr(acc), ptr(bif), s),
    }
    sd.B = B
    for name, call in steps.items():                 # one ordinary pass first: the session exists
        assert call(binding._stream()) == 0, (name, sd.last_error())
    torch.cuda.synchronize()
    for name, call in steps.items():
        g = torch.cuda.CUDAGraph(keep_graph=True)
        before = sd.launch_count()
        with torch.cuda.graph(g):
            assert call(binding._stream()) == 0, (name, sd.last_error())
        assert sd.launch_count() - before == _kernel_nodes(g), name
        del g
    before = sd.launch_count()
    sd.integrity()
    assert sd.launch_count() - before == 2           # red zones, non-finite scan
    sd.close()


@pytest.mark.parametrize("d,f,B,k,attention,layer_gemms", [
    (256, 512, 1, 8, 4, 4),          # both projections inside the attention: a layer's GEMMs are QKV, FFN1 and FFN2
    (256, 448, 1, 8, 4, 4),          # ... where the extra launch of the output projection has no room: a GEMM again while the bit is set
    (256, 512, 40, 20, 4, 6),        # separate launches
])
def test_diag_repeat_adds_the_launches_of_its_class_and_changes_nothing(d, f, B, k, attention, layer_gemms):
    from paper_2203_16487_b200 import binding
    V = 515
    dims = W.ModelDims(d, d // 64, f, V, 1, 2, 128)
    wv, wd = W.make_weights(dims, 5, True), W.make_weights(dims, 6, True)
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=k, max_batch=B, max_src=20, max_tgt=40, bf16=True)
    sd.set_option("debug_checks", 1)
    rng = np.random.default_rng(1)
    src = np.stack([W.zipf_ids(rng, 20, V) for _ in range(B)])
    i32 = dict(dtype=torch.int32, device="cuda")
    draft, acc, bif = torch.randint(4, V, (B, k), **i32), torch.zeros(B, **i32), torch.zeros(B, **i32)
    launches, results = {}, {}
    for bit in (0, 1, 2, 4, 8):
        sd.set_option("diag_repeat", bit)
        sd.encode(src, [20] * B)
        checks = sd.launch_count()
        sd.integrity()
        checks = sd.launch_count() - checks
        before = sd.launch_count()
        sd.verify_raw(draft, 3, 1.0, acc, bif)
        launches[bit] = sd.launch_count() - before - checks
        results[bit] = (sd.debug_row_stats(k), acc.clone(), bif.clone())
    extra = {bit: launches[bit] - launches[0] for bit in (1, 2, 4, 8)}
    norms = launches[0] - attention - layer_gemms - 1 - 2 - (6 if layer_gemms == 6 else 2)      # what is left of the step without the residual GEMMs
    if f == 448:
        assert extra[1] == 2 * attention                     # four attentions and the four output projections they no longer contain
    else:
        assert extra[1] == attention
    assert (extra[2], extra[4], extra[8]) == (norms, layer_gemms, 1)
    for bit in (1, 2, 4, 8):
        if (bit, f) == (1, 448):         # a projection inside the attention and one in a GEMM add in another order: the logits agree as bf16 operands let them
            assert torch.allclose(results[bit][0][..., [0, 4]], results[0][0][..., [0, 4]], atol=2e-2, rtol=1e-2)
        else:
            assert all(torch.equal(a, b) for a, b in zip(results[bit], results[0])), bit
    sd.close()
