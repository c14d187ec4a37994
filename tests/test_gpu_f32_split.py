"""GPU parity of the fp32 relevance and merge (FFMA tiles split over K in a
cluster): every cluster size, shares that end inside a K step, ragged row,
column and text tiles, more critical rows than one compaction window, several
column tiles per cluster, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_25332_gb300 import provip as P
from parity import assert_close_rel, check_merge

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
    (64, 8, (1,)),              # one CTA per cluster, a K step of 8 elements
    (65, 264, (3, 70)),         # clusters of two, shares of 128 and 136
    (130, 520, (64, 0, 65)),    # of four; a sample without text
    (37, 4096, (64,)),          # of eight
    (900, 1096, (33, 90, 128)),
    (40, 136, (1500, 1024)),    # two windows of text rows
])
def test_relevance_f32(N_v, D, tls):
    rng = np.random.default_rng(N_v + D)
    B, T = len(tls), max(tls)
    ev = torch.from_numpy(rng.standard_normal((B, N_v, D)).astype(np.float32))
    et = torch.from_numpy(rng.standard_normal((B, T, D)).astype(np.float32))
    mask = (rng.random((B, T)) < 0.8).astype(np.uint8)
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
        # cosines (at most 1) from fp32 sums: the fp32 path's 1e-5, five times tighter
        assert_close_rel(got, ref, 0.0, f"p N_v={N_v} D={D} tls={tls} [{b}]", atol=2e-6)


@pytest.mark.parametrize("B,N_v,D,keep", [
    (1, 70, 8, 3),       # one column tile, 67 pruned rows
    (2, 300, 264, 65),   # two column tiles, clusters of two
    (1, 577, 4096, 191),
    (3, 400, 520, 399),  # one pruned row, clusters of four
    (8, 800, 512, 200),  # splits of several column tiles
    (2, 50, 64, 50),     # nothing pruned
    (1, 1300, 64, 1100),  # more column tiles than splits
])
def test_merge_f32(B, N_v, D, keep):
    rng = np.random.default_rng(N_v + keep)
    ev = torch.from_numpy(rng.standard_normal((B, N_v, D)).astype(np.float32))
    ev[:, 3] = 0.0
    ev[:, 7] = ev[:, 5]  # exact ties
    keeps = np.stack([np.sort(rng.choice(N_v, keep, replace=False)) for _ in range(B)]).astype(np.int32)
    assign, merged = P.provip_merge(ev.to(DEV), torch.from_numpy(keeps).to(DEV))
    torch.cuda.synchronize()
    for b in range(B):
        Evn = ev[b].double().numpy()
        a_ref, mg_ref = oracle.merge(Evn, keeps[b])
        check_merge(Evn, keeps[b], assign[b].cpu().numpy(), merged[b].double().cpu().numpy(), "f32",
                    f"merge f32 B={B} N_v={N_v} D={D} keep={keep} [{b}]", a_ref,
                    np.setdiff1d(np.arange(N_v), keeps[b]), mg_ref=mg_ref)


def test_merge_bf16_past_the_tensor_core_form():
    """More kept rows than the tensor-core Gram's column ranges hold: the FFMA form on bf16 rows."""
    rng = np.random.default_rng(5)
    N_v, D, keep = 41070, 264, 41000
    ev = torch.from_numpy(rng.standard_normal((1, N_v, D)).astype(np.float32)).to(torch.bfloat16)
    keeps = np.sort(rng.choice(N_v, keep, replace=False)).astype(np.int32)[None]
    assign, merged = P.provip_merge(ev.to(DEV), torch.from_numpy(keeps).to(DEV))
    torch.cuda.synchronize()
    Evn = ev[0].double().numpy()
    a_ref, mg_ref = oracle.merge(Evn, keeps[0])
    check_merge(Evn, keeps[0], assign[0].cpu().numpy(), merged[0].double().cpu().numpy(), "bf16", "merge bf16 FFMA",
                a_ref, np.setdiff1d(np.arange(N_v), keeps[0]), mg_ref=mg_ref)


@pytest.mark.parametrize("tls,T,D", [
    ((64,), 64, 2048),        # one tile, K in two parts of eight shares
    ((65, 40), 65, 2056),     # four tiles, shares that end inside a K step
    ((128, 1, 0), 128, 4096),
    ((20,), 20, 1024),        # shares too short for parts
    ((129,), 129, 4096),      # more text rows than the finish adds parts for
])
def test_critical_rows_f32(tls, T, D):
    rng = np.random.default_rng(T + D)
    # rows whose products stay near 1, so that the softmax is no row's own diagonal
    et = torch.from_numpy((rng.standard_normal((len(tls), T, D)) / D ** 0.5).astype(np.float32))
    for b, t in enumerate(tls):
        et[b, t:] = float("nan")
    mask, r = P.provip_crit_text(et.to(DEV), torch.tensor(tls, dtype=torch.int32, device=DEV), want_r=True)
    torch.cuda.synchronize()
    for b, t in enumerate(tls):
        assert not mask[b, t:].any()
        if t == 0:
            continue
        x = et[b, :t].double()
        ref = torch.softmax(x @ x.T, 1).mean(0).numpy()
        assert_close_rel(r[b, :t].cpu().numpy(), ref, 1e-5, f"r T={T} D={D} [{b}]")
        sure = np.abs(ref - ref.mean()) > 1e-5 * ref.mean()
        got = mask[b, :t].cpu().numpy().astype(bool)
        assert np.array_equal(got[sure], (ref > ref.mean())[sure]) or t == 1
