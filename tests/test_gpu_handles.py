"""Several handles of one process: what a kernel needs of the device is set for the kernel, not for one handle or one launch.
Shared-memory limits belong to a kernel in the whole process, so handles whose launches need different amounts of it are the case to try."""
import threading

import numpy as np
import pytest
import torch

from oracle import specdec_oracle as O
from paper_2203_16487_b200 import workloads as W

pytestmark = pytest.mark.gpu


def _pair(d, H, f, layers, bf16, max_pos=64, V=300):
    dims = W.ModelDims(d, H, f, V, 1, layers, max_pos)
    return dims, W.make_weights(dims, 90 + f, bf16), W.make_weights(dims, 91 + f, bf16)


@pytest.mark.parametrize("bf16", [False, True])
def test_a_later_handle_with_fewer_keys_leaves_the_first_one_alone(bf16):
    """Warp-per-row attention holds a row of scores per warp in shared memory: 3300 keys need 52 KB, 3100 need 49 KB."""
    from paper_2203_16487_b200 import binding
    dims, wv, wd = _pair(32, 4, 32, 1, bf16, max_pos=3400)
    mv = O.model_from(dims, wv, mode="bf16" if bf16 else "pure")
    src = W.zipf_ids(np.random.default_rng(3), 3300, dims.vocab)
    make = lambda n: binding.SpecDec(dims, wv, dims, wd, k_max=4, max_batch=1, max_src=n, max_tgt=8, bf16=bf16)   # noqa: E731
    first, second = make(3300), make(3100)
    first.set_option("attn", 0)
    second.set_option("attn", 0)
    for sd, n in ((second, 3100), (first, 3300)):
        out, m, _ = sd.generate(src[None, :n], [n], [6], 4, 1, 0.0)
        assert out[0, :int(m[0])].cpu().tolist() == O.greedy_decode(mv, src[:n], 6, W.BOS_ID, W.EOS_ID)
    first.close()
    second.close()


@pytest.mark.parametrize("bf16", [False, True])
def test_handles_of_two_host_threads(bf16):
    """Two threads launch the same kernels with different amounts of shared memory (second feed-forward matrix over 1024 and 2048 inputs; fp32:
    128 and 512), without graphs, so that every launch is a launch of the thread's own."""
    from paper_2203_16487_b200 import binding
    handles = []
    for f in ((1024, 2048) if bf16 else (128, 512)):
        dims, wv, wd = _pair(256 if bf16 else 64, 4, f, 6, bf16)
        sd = binding.SpecDec(dims, wv, dims, wd, k_max=8, max_batch=1, max_src=16, max_tgt=24, bf16=bf16)
        sd.set_option("graphs", 0)
        src = W.zipf_ids(np.random.default_rng(f), 12, dims.vocab)
        drafts = torch.arange(10, 18, dtype=torch.int32, device="cuda")[None].contiguous()
        acc, bif = (torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2))
        sd.encode(src[None], [12])
        sd.verify_raw(drafts, 3, 1.0, acc, bif)
        torch.cuda.synchronize()
        handles.append((sd, drafts, acc, bif, (int(acc[0]), int(bif[0]))))
    errors = []
    gate = threading.Barrier(2)

    def work(sd, drafts, acc, bif, want):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                gate.wait(30)
                for i in range(300):
                    sd.verify_raw(drafts, 3, 1.0, acc, bif)
                    if i % 50 == 49:
                        stream.synchronize()
                        assert (int(acc[0]), int(bif[0])) == want, i
        except Exception as e:           # noqa: BLE001 -- reported by the test's thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=h) for h in handles]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for h in handles:
        h[0].close()
