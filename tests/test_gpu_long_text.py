"""GPU parity of the relevance and the critical rows past 128 text rows: block
edges, a narrower last block, one K slice, a partial one, the largest text of
the tensor-core form and the first past it, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_25332_gb300 import provip as P
from parity import assert_close_rel, check_mask_band

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


@pytest.mark.parametrize("N_v,D,T", [(500, 512, 129), (300, 4096, 300), (300, 5120, 129), (300, 8192, 513)])
def test_relevance_of_long_text_is_an_fp32_sums(N_v, D, T):
    """p of random rows against 64 bits: an accumulator is truncated at 16 products of 16
    elements at most before it is added in fp32, a loss of about half a unit of 2^-23 of a
    partial sum each, so some five units of 2^-24 of the sums; eight in the 2-norm of p (FFMA
    sums rounded to nearest over the whole width: 10 at 4096, 17 at 8192)."""
    g = torch.Generator().manual_seed(D + T)
    B = 2
    ev = torch.randn(B, N_v, D, generator=g).to(torch.bfloat16).to(DEV)
    et = (0.02 * torch.randn(B, T, D, generator=g)).to(torch.bfloat16).to(DEV)
    mask = (torch.rand(B, T, generator=g) < 0.4).to(torch.uint8).to(DEV)
    p = P.provip_relevance(ev, et, torch.full((B,), T, dtype=torch.int32, device=DEV), mask).double()
    V, W = ev.double(), et.double()
    cos = (W / W.norm(dim=2, keepdim=True)) @ (V / V.norm(dim=2, keepdim=True)).transpose(1, 2)
    ref = (cos - cos.mean(dim=2, keepdim=True)).masked_fill(mask[:, :, None] == 0, -float("inf")).amax(dim=1)
    assert (p - ref).norm() <= 8 * 2.0 ** -24 * ref.norm()


@pytest.mark.parametrize("N_v,D,T", [(700, 512, 129), (130, 4096, 300), (700, 5120, 300), (97, 8192, 1000), (60, 72, 256)])
def test_norms_of_the_visual_rows_with_long_text(N_v, D, T):
    """1/|v_j|, which the merge reads after the relevance (the first part of its workspace),
    comes from an fp32 sum: slices of 64 products, each to a few roundings that vary from
    slice to slice, added without loss, then a root and a quotient, rounded once each. Two
    units of 2^-24 in the root mean square."""
    g = torch.Generator().manual_seed(D + N_v)
    B = 2
    ev = torch.randn(B, N_v, D, generator=g).to(torch.bfloat16).to(DEV)
    ev[1, 5] = 0
    et = torch.randn(B, T, D, generator=g).to(torch.bfloat16).to(DEV)
    tl = torch.tensor([T, 3], dtype=torch.int32, device=DEV)
    mask = torch.ones(B, T, dtype=torch.uint8, device=DEV)
    L = P.lib()
    ws = P.workspace(L.provip_relevance_workspace_size(B, N_v, D, T), torch.device(DEV))
    p = torch.empty(B, N_v, dtype=torch.float32, device=DEV)
    rc = L.provip_relevance(P._ptr(ev), B, N_v, D, P._ptr(et), P._i32(tl), T, P._u8(mask), P.BF16, P._ptr(p), P._ptr(ws),
                            ws.numel(), P._stream(ev.device))
    assert rc == 0
    torch.cuda.synchronize()
    inv = ws[:4 * B * N_v].view(torch.float32).view(B, N_v).double()
    assert inv[1, 5] == 0
    norm = ev.double().norm(dim=2)
    rel = (inv * norm - 1)[norm > 0]
    assert rel.square().mean().sqrt() <= 2 * 2.0 ** -24


@pytest.mark.parametrize("dtype,D,tls", [
    ("bf16", 64, (1, 5, 128)),               # one K slice: a cluster of one CTA
    ("bf16", 264, (17, 0, 33)),              # five slices over four CTAs
    ("bf16", 520, (100,)),                   # nine slices over eight CTAs, a partial last one
    ("bf16", 4096, (96, 128, 31)),           # 8 CTAs of two accumulators
    ("bf16", 1024, tuple(range(100, 140))),  # 2 x 2 tiles, 4 CTAs of four accumulators
    ("bf16", 1024, tuple(range(60, 90))),    # one tile, 4 CTAs of four accumulators
    ("bf16", 72, (129, 257, 1)),
    ("bf16", 256, (513, 40)),                # past the columns held in registers
    ("f32", 64, (1, 128, 40)),
    ("f32", 264, (129, 511)),
    ("f32", 64, (700, 513)),
])
def test_critical_rows(dtype, D, tls):
    rng = np.random.default_rng(D + len(tls))
    B, T = len(tls), max(tls)
    # text logits at the scale of LLM token embeddings: a smooth softmax
    et = torch.from_numpy((rng.standard_normal((B, T, D)) * 0.25 / D ** 0.25).astype(np.float32))
    et = et.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    for b, t in enumerate(tls):
        et[b, t:] = float("nan")
    mask, r = P.provip_crit_text(et.to(DEV), torch.tensor(tls, dtype=torch.int32, device=DEV), want_r=True)
    torch.cuda.synchronize()
    for b, t in enumerate(tls):
        m, rr = mask[b].cpu().numpy(), r[b].cpu().numpy()
        assert not m[t:].any() and not rr[t:].any()
        if t == 0:
            continue
        r_ref, _ = oracle.crit_text(et[b, :t].double().numpy())
        # logits of order 1 in fp32 sums (their exponentials a few ulp off)
        assert_close_rel(rr[:t], r_ref, 1e-5, f"r {dtype} D={D} tls={tls} [{b}]")
        check_mask_band(m[:t], r_ref, 1e-5, f"T {dtype} D={D} tls={tls} [{b}]")
