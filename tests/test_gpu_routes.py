"""Which kernel serves a launch, read off the kernel nodes of a captured step: the rules that were set by measuring both sides, at their edges."""
import ctypes as C
import re

import numpy as np
import pytest
import torch

from paper_2203_16487_b200 import workloads as W

pytestmark = pytest.mark.gpu

CU_GRAPH_NODE_TYPE_KERNEL = 0
RESID = "2"                                           # (the epilogue that adds to the residual stream)


class KernelNode(C.Structure):                        # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p)] + [(n, C.c_uint) for n in ("gx", "gy", "gz", "bx", "by", "bz", "smem")] + \
               [(n, C.c_void_p) for n in ("params", "extra", "kern", "ctx")]


def _kernels(graph):
    """Names with template arguments, as k_rows<2,0,1,8,2,1,8>, of the graph's kernel nodes."""
    cu, g, n = C.CDLL("libcuda.so.1"), C.c_void_p(graph.raw_cuda_graph()), C.c_size_t()
    assert cu.cuGraphGetNodes(g, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, C.byref(n)) == 0
    names = []
    for node in nodes:
        t, p, name = C.c_int(), KernelNode(), C.c_char_p()
        assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(t)) == 0
        if t.value != CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)) == 0
        assert (cu.cuFuncGetName(C.byref(name), C.c_void_p(p.func)) if p.func else cu.cuKernelGetName(C.byref(name), C.c_void_p(p.kern))) == 0
        m = re.match(r"_ZN?(?:2sd)?\d+(k_[a-z0-9_]+?)(?:I(.*?)E+v.*|E?P.*|$)", name.value.decode())
        args = re.findall(r"L[ib](\d+)E", m.group(2) + "E") if m and m.group(2) else []
        names.append(f"{m.group(1)}<{','.join(args)}>" if m else name.value.decode())
    return names


def launched(call):
    """Names of the kernels that a step call launches (a handle without graphs: its launches go into the capture)."""
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    return _kernels(g)


def _step(dims, step, B, k, S):
    from paper_2203_16487_b200 import binding
    wv, wd = W.make_weights(dims, 5, True), W.make_weights(dims, 6, True)
    sd = binding.SpecDec(dims, wv, dims, wd, k_max=max(k, 1), max_batch=B, max_src=S, max_tgt=40, bf16=True)
    sd.set_option("graphs", 0)                        # the step calls launch into the capture themselves
    rng = np.random.default_rng(1)
    src = torch.from_numpy(np.stack([W.zipf_ids(rng, S, dims.vocab) for _ in range(B)])).cuda()
    i32 = dict(dtype=torch.int32, device="cuda")
    lens, draft, acc, bif = torch.full((B,), S, **i32), torch.zeros((B, max(k, 1)), **i32), torch.zeros(B, **i32), torch.zeros(B, **i32)
    lib, ptr = sd._lib, binding._ptr
    calls = {
        "encode": lambda s: lib.specdec_encode(sd._h, ptr(src), ptr(lens), None, B, S, s),
        "verify": lambda s: lib.specdec_verify(sd._h, ptr(draft), k, 3, 1.0, ptr(acc), ptr(bif), s),
    }
    sd.B = B
    for name in dict.fromkeys(("encode", step)):      # an ordinary pass first: the session exists
        assert calls[name](binding._stream()) == 0, sd.last_error()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        assert calls[step](binding._stream()) == 0, sd.last_error()
    names = _kernels(g)
    del g
    sd.close()
    return names


def _resid(names):
    """The launches that add to the residual stream, in order."""
    return [n for n in names if n.startswith("k_gemm_tc_splitk") or re.match(rf"k_(rows|gemm_tc)<{RESID},", n)]


# One decoder layer: output projections of both attentions, then FFN2.
@pytest.mark.parametrize("d,f,B,k,ffn2", [
    (512, 2112, 8, 15, "k_rows"),           # 128 rows.  K = 2112 is 33 K blocks, which no two or four slices share equally:
    (512, 2112, 10, 12, "k_rows"),          # 130 rows: the few-rows kernel goes on to its own limit
    (512, 2112, 11, 15, "k_rows"),          # 176 rows: the last
    (512, 2112, 12, 15, "k_gemm_tc<"),      # 192 rows: whole tiles
    (512, 2048, 8, 15, "k_rows"),           # 128 rows
    (512, 2048, 10, 12, "k_gemm_tc_splitk"),
    (512, 2176, 10, 12, "k_gemm_tc_splitk"),
    (768, 2112, 8, 9, "k_rows"),            # 80 rows
    (768, 2112, 8, 11, "k_rows"),           # 96 rows
    (768, 2112, 7, 13, "k_gemm_tc<"),       # 98 rows
    (768, 3072, 8, 10, "k_gemm_tc_splitk"),  # 88 rows
])
def test_ffn2_leaves_the_few_rows_kernel_for_split_tiles_only(d, f, B, k, ffn2):
    names = _step(W.ModelDims(d, d // 64, f, 515, 1, 1, 64), "verify", B, k, 12)
    assert _resid(names)[-1].startswith(ffn2), names


# Two equal encoders of one layer each: output projection, then FFN2, of each.
@pytest.mark.parametrize("d,B,S,out", [
    (512, 8, 9, "k_rows<2,0,1,"),               # 72 rows: the last few-rows tiles
    (512, 1, 73, "k_rows<2,0,1,8,2,1,8>"),      # 16-row tiles with the weights as fragments, from here on
    (512, 8, 12, "k_rows<2,0,1,8,2,1,8>"),      # 96 rows
    (512, 1, 97, "k_rows<2,0,1,8,2,1,8>"),
    (512, 16, 16, "k_rows<2,0,1,8,2,1,8>"),     # 256 rows: the last
    (512, 1, 257, "k_rows<2,0,2,8,2,1,8>"),     # 32-row tiles
    (512, 20, 16, "k_rows<2,0,2,8,2,1,8>"),     # 320 rows: the last
    (512, 3, 107, "k_gemm_tc<2,"),              # 321 rows
    (512, 36, 16, "k_gemm_tc<2,"),              # 576 rows
    (768, 4, 10, "k_rows<2,0,1,"),              # 40 rows
    (768, 1, 41, "k_rows<2,0,1,4,1,1,6>"),      # 41 rows
    (768, 2, 48, "k_rows<2,0,1,4,1,1,6>"),      # 96 rows: the last at this width
])
def test_output_projections_of_the_encoders(d, B, S, out):
    names = _resid(_step(W.ModelDims(d, d // 64, 4 * d, 515, 1, 1, 320), "encode", B, 0, S))
    assert len(names) == 4 and names[0].startswith(out) and names[2].startswith(out), names


# The projections of 32-row tiles (QKV, FFN1, wider output projections) of encoders with 64- and with 32-wide heads.
@pytest.mark.parametrize("d,B,S", [(512, 8, 12), (512, 10, 16), (512, 14, 16), (512, 20, 16), (768, 12, 16)])       # 96, 160, 224, 320, 192 rows
def test_32_row_tiles_of_the_encoders_go_with_tile_attention(d, B, S):
    wide, narrow = (sum(n.startswith("k_rows<") and ",0,2,8,2,1," in n for n in _step(W.ModelDims(d, d // dh, 4 * d, 515, 1, 1, 128), "encode", B, 0, S))
                    for dh in (64, 32))
    assert wide > 0 and narrow == 0


@pytest.mark.parametrize("d,f,split", [
    (512, 1024, False),
    (512, 1664, False),
    (512, 1792, True),                      # 512 columns: the shortest reduction that gains
    (512, 2048, True),
    (1024, 2048, True),                     # (output projections: K = 1024)
])
def test_two_slices_of_128_columns_are_for_long_reductions(d, f, split):
    B, k = (48, 25) if d == 512 else (40, 25)
    names = _resid(_step(W.ModelDims(d, d // 64, f, 515, 1, 1, 128), "verify", B, k, 12))
    assert [n.startswith("k_gemm_tc_splitk<2,128,128>") for n in names] == [False, False, split], names


# One decoder layer: whether the self-attention goes on to its output projection, the cross-attention projects its queries, and goes on to its output projection.
@pytest.mark.parametrize("d,B,k,S,self_out,cross_q,cross_out", [
    (512, 1, 3, 12, 0, 1, 0),               # 4 rows: too few to gain
    (256, 1, 4, 12, 1, 1, 1),               # 5 rows
    (512, 1, 15, 128, 1, 1, 1),             # eight heads, 8 CTAs; as many keys as fit beside the queries' projection
    (512, 1, 15, 129, 1, 1, 0),             # a key more
    (512, 1, 16, 128, 0, 1, 1),             # 16 CTAs
    (512, 2, 15, 128, 0, 1, 1),
    (512, 1, 32, 128, 0, 1, 0),             # 24 CTAs
    (256, 2, 23, 128, 1, 1, 1),             # four heads, 48 rows
    (256, 1, 48, 128, 1, 1, 0),             # 49 rows
    (256, 8, 16, 12, 1, 1, 0),              # 64 CTAs
    (256, 9, 16, 12, 0, 1, 0),              # 72 CTAs
])
def test_projections_inside_the_attention(d, B, k, S, self_out, cross_q, cross_out):
    names = _step(W.ModelDims(d, d // 64, 2 * d, 515, 1, 1, 256), "verify", B, k, S)
    (_, s_out), (c_q, c_out) = ([int(v) > 0 for v in n[:-1].split(",")[-2:]] for n in names if n.startswith("k_attn<"))
    assert (s_out, c_q, c_out) == (self_out, cross_q, cross_out), names


# One layer: the attention kernels of a verify step (self, cross) or of the two encoders.  Over at most 128 keys the key groups share their probabilities (the sixth argument), four
# groups from five queries on.
@pytest.mark.parametrize("step,d,k,S,kernels", [
    ("verify", 128, 4, 128, "1,1,4,32,3,1,0,0 0,1,4,32,3,1,0,0"),       # 5 queries
    ("verify", 128, 4, 129, "1,1,4,32,3,1,0,0 0,1,4,32,3,0,0,0"),       # a key more
    ("verify", 128, 3, 128, "1,1,4,32,3,0,0,0 0,1,4,32,3,0,0,0"),       # 4 queries
    ("verify", 512, 3, 128, "1,1,4,32,3,0,0,0 0,1,8,16,3,1,4,0"),       # eight groups share from one query on
    ("verify", 512, 0, 128, "1,1,4,32,3,0,0,0 0,1,8,16,3,1,4,0"),
    ("verify", 512, 3, 129, "1,1,4,32,3,0,0,0 0,1,8,32,2,0,4,0"),
    ("verify", 256, 4, 128, "1,1,8,16,3,1,0,4 0,1,8,16,3,1,2,4"),
    ("verify", 256, 4, 129, "1,1,8,16,3,1,0,4 0,1,8,32,2,0,2,0"),       # no room for both projections beside a second block
    ("verify", 512, 15, 128, "1,1,8,16,3,1,0,8 0,1,8,16,3,1,4,8"),
    ("verify", 768, 4, 128, "1,1,4,32,3,1,0,0 0,1,8,16,3,1,6,0"),
    ("verify", 768, 4, 129, "1,1,4,32,3,1,0,0 0,1,8,16,3,0,6,0"),
    ("encode", 128, 0, 128, "0,1,4,32,3,1,0,0 0,1,4,32,3,1,0,0"),
    ("encode", 128, 0, 129, "0,1,4,32,3,0,0,0 0,1,4,32,3,0,0,0"),
    ("encode", 128, 0, 5, "0,1,4,32,3,1,0,0 0,1,4,32,3,1,0,0"),
    ("encode", 128, 0, 4, "0,1,4,32,3,0,0,0 0,1,4,32,3,0,0,0"),
    ("encode", 256, 0, 128, "0,1,8,16,3,1,0,4 0,1,8,16,3,1,0,4"),
    ("encode", 256, 0, 129, "0,1,8,16,3,0,0,4 0,1,8,16,3,0,0,4"),
])
def test_key_groups_share_probabilities_over_one_block(step, d, k, S, kernels):
    names = _step(W.ModelDims(d, d // 64, 2 * d, 515, 1, 1, 256), step, 1, k, S)
    assert [n for n in names if n.startswith("k_attn<")] == [f"k_attn<{a}>" for a in kernels.split()], names
