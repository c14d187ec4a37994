"""Merge Gram on pairs of SMs with 256-row groups: the tile plan and the choice of
the form (host logic compiled from the library's source, on the CPU), and both
forms on the GPU with ragged groups and ranges against the oracle."""
import os
import subprocess

import numpy as np
import pytest
import torch

from test_merge_plan import HERE, _nvcc

# (B, N_v, keep, D), the form that the plan takes on 152 SMs
FORMS = [((16, 576, 288, 4096), 1), ((32, 576, 192, 5120), 1), ((4, 1443, 481, 4096), 1), ((1, 40, 3, 64), 1),
         ((8, 2880, 960, 4096), 2), ((1, 9216, 2304, 3584), 2), ((24, 1320, 500, 2048), 2)]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cc = _nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("plan") / "merge_half_plan_check")
    r = subprocess.run([cc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + os.path.join(os.path.dirname(HERE), "include"),
                        os.path.join(HERE, "merge_half_plan_check.cu"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return out


def _lines(checker, shapes):
    r = subprocess.run([checker, *(str(v) for s in shapes for v in s)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.splitlines()


def test_chosen_forms(checker):
    assert _lines(checker, [(*s, 152) for s, _ in FORMS]) == [f"ok {f}" for _, f in FORMS]


def test_half_plans_of_random_shapes(checker):
    rng = np.random.default_rng(7)
    shapes = []
    for _ in range(60):
        N_v = int(rng.integers(2, 6000))
        shapes.append((int(rng.integers(1, 24)), N_v, int(rng.integers(1, min(N_v - 1, 4096) + 1)),
                       8 * int(rng.integers(1, 600)), 2 * int(rng.integers(1, 90))))
    shapes += [(3, 257, 1, 64, 152), (3, 258, 1, 64, 152), (2, 513, 256, 64, 152), (2, 514, 257, 64, 152)]
    assert len(_lines(checker, shapes)) == len(shapes)


@pytest.mark.gpu
@pytest.mark.parametrize("B,N_v,D,keep,form", [
    (2, 257, 64, 1, 1),      # one group of exactly 256 rows
    (2, 258, 72, 1, 1),      # a second group of one row
    (3, 700, 136, 257, 1),   # 443 pruned rows, two ranges, a partial last K slice
    (1, 130, 1032, 100, 1),  # 30 pruned rows, 17 slices through six stages
    (26, 1500, 512, 300, 2),  # 512-row groups, two tiles per pair of SMs, the last group one half
])
def test_merge_with_either_form(checker, B, N_v, D, keep, form):
    import __graft_entry__
    import oracle
    from paper_2608_25332_gb300 import provip as P
    from parity import check_merge
    __graft_entry__.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert _lines(checker, [(B, N_v, keep, D, sms)]) == [f"ok {form}"]
    rng = np.random.default_rng(N_v + keep)
    ev = torch.from_numpy(rng.standard_normal((B, N_v, D)).astype(np.float32)).to(torch.bfloat16)
    ev[:, 7] = ev[:, 5]  # exact ties
    keeps = np.stack([np.sort(rng.choice(N_v, keep, replace=False)) for _ in range(B)]).astype(np.int32)
    assign, merged = P.provip_merge(ev.to("cuda:0"), torch.from_numpy(keeps).to("cuda:0"))
    torch.cuda.synchronize()
    for b in {0, B // 2, B - 1}:
        Evn = ev[b].double().numpy()
        a_ref, mg_ref = oracle.merge(Evn, keeps[b])
        check_merge(Evn, keeps[b], assign[b].cpu().numpy(), merged[b].double().cpu().numpy(), "bf16",
                    f"merge B={B} N_v={N_v} D={D} keep={keep} [{b}]", a_ref, np.setdiff1d(np.arange(N_v), keeps[b]),
                    mg_ref=mg_ref)
    rc, bits = P.provip_device_status(clear=True)
    assert rc == 0 and bits == 0
