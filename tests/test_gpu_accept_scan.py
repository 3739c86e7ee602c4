"""The acceptance rule on a caller's logits against the oracle, at the sizes where the launch rule and the row walk change:
one CTA or clusters of 8 / 16 per sequence, rows that are not a multiple of four columns (unaligned row starts, heads and
tails), decisions on the first and the last row of a group and beyond the first group, exact ties, rows of -inf."""
import numpy as np
import pytest
import torch

from oracle import specdec_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,k,V", [(3, 40, 5), (2, 1, 4096), (16, 17, 4097), (17, 9, 5003), (33, 8, 4099), (5, 33, 50265)])
def test_accept_scan_edges(B, k, V):
    from paper_2203_16487_b200 import binding
    rng = np.random.default_rng(B * 1000 + k)
    logits = (rng.standard_normal((B, k + 1, V)) * 3).astype(np.float32)
    drafts = logits.argmax(axis=2)[:, :k].astype(np.int32)
    stop = [(0, 7, 8, 15, 16, 24, 31, 32)[b % 8] for b in range(B)]           # first rejected row of each sequence, where k reaches it
    for b in range(B):
        if b != 1 and stop[b] < k:
            drafts[b, stop[b]] = int(np.argmin(logits[b, stop[b]]))
    logits[0, 0, [0, V - 1]] = logits[0, 0].max() + 1.0                       # a tie between the first and the last column
    logits[-1, -1] = -np.inf
    logits[-1, -1, V // 2] = -5.0
    if B > 2:
        drafts[2, 0] = V + 3                                                 # not a token: rejected
    lg, dr = torch.from_numpy(logits).cuda(), torch.from_numpy(drafts).cuda()
    for beta, tau in ((3, 1.0), (1, 0.0)):
        # (other work holds SMs meanwhile, so that the CTAs of a cluster need not begin together)
        other = torch.cuda.Stream()
        with torch.cuda.stream(other):
            busy = torch.ones((2048, 2048), device="cuda")
            for _ in range(8):
                busy = busy @ busy * 1e-4
        a, t = binding.accept_scan(lg, dr, beta, tau)
        for b in range(B):
            row = drafts[b].tolist()
            if not 0 <= row[0] < V:
                want = (0, int(logits[b, 0].argmax()))
            else:
                want = O.verify(logits[b], row, beta, tau)
            assert (int(a[b]), int(t[b])) == want, (b, beta, tau)
