"""Pre-LLM pass with the critical rows first on the stream and from the side stream: the
mask and p of back-to-back passes on one workspace must be the bits of the separate
calls."""
import pytest
import torch

import __graft_entry__

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("B,N_v,N_t,D,keep", [
    (13, 100, 40, 512, 30),    # 104 CTAs: the side stream
    (15, 100, 40, 512, 30),    # 120 CTAs of clusters of 8: first on the stream
    (15, 560, 40, 512, 30),    # the same, but a relevance CTA fits beside each on nearly every SM: the side stream
    (15, 560, 128, 512, 30),   # one that does not fit: first
    (20, 300, 128, 256, 100),  # clusters of 4 (as many K slices): 80 CTAs, the side stream
    (29, 257, 128, 264, 64),   # clusters of 4: 116 CTAs, first; a ragged last K slice and visual tile
    (120, 40, 7, 64, 9),       # one K slice, one CTA a sample: first
    (140, 40, 7, 64, 9),       # the same on nearly every SM: the side stream
    (64, 70, 128, 256, 20),    # clusters of 4, 512 columns of tensor memory each: 256 CTAs, more than SMs; first
])
def test_pass_gives_the_bits_of_separate_calls(B, N_v, N_t, D, keep):
    __graft_entry__.build()
    from paper_2608_25332_gb300 import provip as P
    g = torch.Generator().manual_seed(B)
    sets = []
    for _ in range(3):
        ev = torch.randn(B, N_v, D, generator=g).to(torch.bfloat16).to(DEV)
        et = (0.1 * torch.randn(B, N_t, D, generator=g)).to(torch.bfloat16).to(DEV)
        tl = torch.randint(0, N_t + 1, (B,), generator=g, dtype=torch.int32).to(DEV)
        sets.append((ev, et, tl))
    want = []
    for ev, et, tl in sets:
        mask = P.provip_crit_text(et, tl)
        torch.cuda.synchronize()
        p = P.provip_relevance(ev, et, tl, mask)
        torch.cuda.synchronize()
        want.append((mask.clone(), p.clone()))
    ws = P.workspace(P.lib().provip_similarity_reduce_workspace_size(B, N_v, D, N_t, keep), torch.device(DEV))
    for _ in range(2):
        got = [P.provip_similarity_reduce(ev, et, tl, keep, want_merged=True, ws=ws) for ev, et, tl in sets]  # no sync between
        torch.cuda.synchronize()
        for (mask, p), r in zip(want, got):
            assert torch.equal(mask, r["mask"]) and torch.equal(p, r["p"])
    rc, bits = P.provip_device_status(clear=True)
    assert rc == 0 and bits == 0
