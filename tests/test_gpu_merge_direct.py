"""Merge Gram reading its rows where they lie: when the plan chooses it (host logic
compiled from the library's source, on the CPU), and ragged groups, ranges, widths
and deals against the oracle on the GPU."""
import os
import subprocess

import numpy as np
import pytest
import torch

from test_merge_plan import HERE, _nvcc

# (B, N_v, keep, D) on 152 SMs
FORMS = [((32, 576, 192, 5120), "1 direct"), ((8, 2880, 960, 4096), "2 direct"), ((4, 1443, 481, 4096), "1 direct"),
         ((1, 9216, 2304, 3584), "2 copy"), ((1, 576, 144, 4096), "1 copy")]


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cc = _nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("form") / "merge_form_check")
    r = subprocess.run([cc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + os.path.join(os.path.dirname(HERE), "include"),
                        os.path.join(HERE, "merge_form_check.cu"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return out


def _forms(checker, shapes):
    r = subprocess.run([checker, *(str(v) for s in shapes for v in s)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.splitlines()


def test_chosen_forms(checker):
    assert _forms(checker, [(*s, 152) for s, _ in FORMS]) == [f for _, f in FORMS]


def _search(checker, shapes):
    r = subprocess.run([checker, "search", *(str(v) for s in shapes for v in s)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return [float(line.split()[1]) for line in r.stdout.splitlines()]


def test_plans_are_the_full_searchs(checker):
    """Both group sizes' plans are those of a search that deals every candidate's tiles."""
    rng = np.random.default_rng(11)
    shapes = [(*s, 152) for s, _ in FORMS] + [(3, 257, 1, 64, 152), (2, 513, 256, 64, 152), (1, 600, 1, 64, 2)]
    for _ in range(60):
        N_v = int(rng.integers(2, 6000))
        shapes.append((int(rng.integers(1, 40)), N_v, int(rng.integers(1, min(N_v - 1, 5000) + 1)),
                       8 * int(rng.integers(1, 600)), 2 * int(rng.integers(1, 90))))
    assert len(_search(checker, shapes)) == len(shapes)


def test_a_new_shape_costs_less_than_one_full_search(checker):
    """Host time of a shape not seen before against that of one search that deals every
    candidate's tiles (measured 0.02 to 0.4)."""
    shapes = [(8, 2880, 960, 4096, 152), (1, 9216, 2304, 3584, 152), (4, 1443, 481, 4096, 152), (64, 2880, 960, 4096, 152)]
    assert max(_search(checker, shapes)) < 1


@pytest.mark.gpu
@pytest.mark.parametrize("B,N_v,D,keep,halves", [
    (32, 258, 64, 1, 1),      # a second group of one row; one kept row; one K slice
    (32, 420, 72, 40, 1),     # a width that ends inside the second K slice
    (90, 280, 136, 24, 1),    # two tiles per pair of SMs, groups of exactly 256 rows
    (40, 450, 520, 257, 1),   # nine slices through six stages, two ranges, a ragged last group
    (26, 1500, 512, 300, 2),  # 512-row groups, the last one half
])
def test_merge_reading_rows_in_place(checker, B, N_v, D, keep, halves):
    import __graft_entry__
    import oracle
    from paper_2608_25332_gb300 import provip as P
    from parity import check_merge
    __graft_entry__.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert _forms(checker, [(B, N_v, keep, D, sms)]) == [f"{halves} direct"]
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
