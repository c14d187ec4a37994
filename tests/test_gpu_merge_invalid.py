"""The merge given a keep_idx with repeated, descending and out-of-range entries: the call
reports it in the device status, and every row, those that such a list leaves over
included, gets a position of the list, whatever the workspace held before."""
import numpy as np
import pytest
import torch

from paper_2608_25332_gb300 import provip as P

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _merge(ev, keeps):
    B, N_v, D = ev.shape
    keep = keeps.shape[1]
    L = P.lib()
    ws = P.workspace(L.provip_merge_workspace_size(B, N_v, D, keep), torch.device(DEV))
    ws.fill_(0x3D)  # as positions far past the list, as cosines 0.046
    assign = torch.empty(B, N_v, dtype=torch.int32, device=DEV)
    merged = torch.empty(B, keep, D, dtype=ev.dtype, device=DEV)
    k = torch.from_numpy(keeps).to(DEV)
    rc = L.provip_merge(P._ptr(ev), B, N_v, D, P._i32(k), keep, P._dtype_code(ev), P._ptr(assign), P._ptr(merged),
                        P._ptr(ws), ws.numel(), P._stream(ev.device))
    assert rc == 0
    rc, bits = P.provip_device_status(clear=True)
    assert rc != 0 and bits == P.DEVSTAT_BAD_ARG
    assert torch.isfinite(merged).all()
    return assign.cpu().numpy()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("N_v,keep,bad", [(300, 5, 3), (300, 90, 80), (140, 139, 9), (70, 70, 6)])
def test_rows_left_over_by_an_invalid_list(dtype, N_v, keep, bad):
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(N_v + keep)
    B, D = 2, 256
    keeps = np.stack([np.sort(rng.choice(N_v, keep, replace=False)) for _ in range(B)]).astype(np.int32)
    for b in range(B):
        for i, q in enumerate(rng.choice(np.arange(1, keep), bad, replace=False)):
            keeps[b, q] = (keeps[b, q - 1], N_v + 7, -3)[i % 3]
    # every row near one of the list's rows, so that its nearest one is clear
    ev = rng.standard_normal((B, N_v, D)).astype(np.float32)
    for b in range(B):
        rows = keeps[b][(keeps[b] >= 0) & (keeps[b] < N_v)]
        near = rng.choice(rows, N_v)
        near[rows] = rows
        ev[b] = ev[b, near] + 0.05 * ev[b]
    ev = torch.from_numpy(ev).to(dtype)
    assign = _merge(ev.to(DEV), keeps)
    assert assign.min() >= 0 and assign.max() < keep
    if dtype == torch.float32:  # the FFMA Gram takes every row that is not kept
        for b in range(B):
            X = ev[b].double().numpy()
            inside = (keeps[b] >= 0) & (keeps[b] < N_v)
            K = np.where(inside[:, None], X[np.where(inside, keeps[b], 0)], 0.0)
            cos = X @ (K / np.maximum(np.linalg.norm(K, axis=1, keepdims=True), 1e-30)).T
            got = cos[np.arange(N_v), assign[b]]
            assert np.all(got >= cos.max(axis=1) - 1e-4 * np.linalg.norm(X, axis=1))
