"""GPU parity of the relevance and the critical rows past 128 text rows: block
edges, a narrower last block, one K slice, a partial one, the largest text of
the tensor-core form and the first past it, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_25332_gb300 import provip as P
from parity import assert_close_rel

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__
    __graft_entry__.build()
    yield
    rc, bits = P.provip_device_status(clear=True)
    assert rc == 0 and bits == 0, f"device status {rc} {bits}"


@pytest.mark.parametrize("N_v,D,tls", [
    (131, 64, (129, 1)),        # one K slice: the second accumulator is never written
    (200, 128, (144, 100)),     # two equal blocks
    (97, 200, (145, 145)),      # ten 16-row groups in blocks of 80
    (300, 1096, (256, 0, 130)),  # a sample without text, a partial last K slice
    (64, 136, (272, 271)),      # three blocks, the last one narrower
    (1000, 264, (513,)),
    (70, 64, (4096,)),
    (70, 64, (4097,)),          # past the tensor-core form
])
def test_relevance_of_long_text(N_v, D, tls):
    rng = np.random.default_rng(N_v + D)
    B, T = len(tls), max(tls)
    ev = torch.from_numpy(rng.standard_normal((B, N_v, D)).astype(np.float32)).to(torch.bfloat16)
    et = torch.from_numpy(rng.standard_normal((B, T, D)).astype(np.float32)).to(torch.bfloat16)
    mask = (rng.random((B, T)) < 0.5).astype(np.uint8)
    for b, t in enumerate(tls):
        et[b, t:] = float("nan")
        if t:
            mask[b, t - 1] = 1
    p = P.provip_relevance(ev.to(DEV), et.to(DEV), torch.tensor(tls, dtype=torch.int32, device=DEV),
                           torch.from_numpy(mask).to(DEV))
    torch.cuda.synchronize()
    for b, t in enumerate(tls):
        got = p[b].cpu().numpy()
        if t == 0:
            assert np.all(np.isneginf(got))
            continue
        ref = oracle.relevance(et[b, :t].double().numpy(), mask[b, :t], ev[b].double().numpy())
        # fp32 sums of at most 1096 exact products: far inside the pass's 2e-3
        assert_close_rel(got, ref, 0.0, f"p N_v={N_v} D={D} tls={tls} [{b}]", atol=1e-5)
