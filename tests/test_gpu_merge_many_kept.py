"""GPU parity of the merge around the number of kept rows up to which the counting sort
keeps its counters in shared memory: the last one that does, the first that does not,
and 6144, where the counters alone fill 48 KiB."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_25332_gb300 import provip as P
from parity import check_merge

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("keep", [6128, 6129, 6144, 6145])
def test_merge_with_thousands_of_kept_rows(keep):
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(keep)
    B, N_v, D = 2, keep + 61, 16
    Ev = rng.standard_normal((B, N_v, D)).astype(np.float32)
    keeps = np.stack([np.sort(rng.choice(N_v, keep, replace=False)) for _ in range(B)]).astype(np.int32)
    assign, merged = P.provip_merge(torch.from_numpy(Ev).to(DEV), torch.from_numpy(keeps).to(DEV))
    torch.cuda.synchronize()
    for b in range(B):
        Evn = Ev[b].astype(np.float64)
        a_ref, mg_ref = oracle.merge(Evn, keeps[b])
        check_merge(Evn, keeps[b], assign[b].cpu().numpy(), merged[b].cpu().numpy().astype(np.float64), "f32",
                    f"keep={keep} [{b}]", a_ref, np.setdiff1d(np.arange(N_v), keeps[b]), mg_ref=mg_ref)
    rc, bits = P.provip_device_status(clear=True)
    assert rc == 0 and bits == 0
