"""GPU parity of the merge's means when some centroids gather many rows (their
own CTAs, a column slice each): member counts at the limit between the two
paths and past one window of the ordering bitmap, rows of every configuration
and of a partial last slice, against the oracle."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_25332_gb300 import provip as P
from parity import check_merge

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__
    __graft_entry__.build()
    yield
    rc, bits = P.provip_device_status(clear=True)
    assert rc == 0 and bits == 0, f"device status {rc} {bits}"


@pytest.mark.parametrize("dtype,D,B", [("bf16", 64, 3), ("bf16", 1040, 2), ("bf16", 4096, 1), ("bf16", 4104, 1),
                                       ("f32", 200, 2), ("f32", 2048, 1), ("f32", 2056, 1)])
def test_merge_means_of_long_centroids(dtype, D, B):
    """Groups of 16, 17, 1 and 1100 rows (the kept one included) around well
    separated directions, scattered over the sample; N_v spans two windows."""
    sizes = (16, 17, 1, 1100, 12, 40)
    rng = np.random.default_rng(D)
    N_v = sum(sizes)
    Ev = np.empty((B, N_v, D), np.float32)
    keeps = np.empty((B, len(sizes)), np.int32)
    for b in range(B):
        place = rng.permutation(N_v)
        o = 0
        for n in sizes:
            c = rng.standard_normal(D)
            rows = place[o:o + n]
            Ev[b, rows] = c + 0.3 * rng.standard_normal((n, D))
            o += n
        heads = [place[sum(sizes[:i])] for i in range(len(sizes))]
        keeps[b] = np.sort(heads)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    ev = torch.from_numpy(Ev).to(td)
    assign, merged = P.provip_merge(ev.to(DEV), torch.from_numpy(keeps).to(DEV))
    torch.cuda.synchronize()
    Evn = ev.float().numpy().astype(np.float64)
    for b in range(B):
        a_ref, mg_ref = oracle.merge(Evn[b], keeps[b])
        assert sorted(np.bincount(a_ref, minlength=len(sizes)).tolist()) == sorted(sizes)
        check_merge(Evn[b], keeps[b], assign[b].cpu().numpy(), merged[b].float().cpu().numpy().astype(np.float64),
                    dtype, f"long centroids {dtype} D={D} [{b}]", a_ref,
                    np.setdiff1d(np.arange(N_v), keeps[b]), mg_ref=mg_ref)


@pytest.mark.parametrize("keep", [2, 40])
@pytest.mark.parametrize("D", [264, 2056])
def test_fp32_means_of_huge_and_non_finite_values(keep, D):
    """fp32 sums that leave fp32's range, cancel, or meet infinities and NaN give
    the means that double sums give (the GPU's own member sets, both paths)."""
    rng = np.random.default_rng(D + keep)
    N_v = 80
    Ev = rng.standard_normal((1, N_v, D)).astype(np.float32)
    Ev[0, :, 0] = 3.0e38                      # the sum overflows fp32, the mean does not
    Ev[0, :, 1] = np.where(np.arange(N_v) % 2, 3.0e38, -3.0e38)
    Ev[0, 9, 2] = np.inf
    Ev[0, 9, 3], Ev[0, 10, 3] = np.inf, -np.inf
    Ev[0, 11, 4] = np.nan
    Ev[0, :, 5] = 1e-40                       # subnormal
    Ev[0, :, 6] = 1e30 * rng.standard_normal(N_v)
    keeps = np.sort(rng.choice(N_v, keep, replace=False)).astype(np.int32)[None]
    assign, merged = P.provip_merge(torch.from_numpy(Ev).to(DEV), torch.from_numpy(keeps).to(DEV))
    torch.cuda.synchronize()
    a = assign[0].cpu().numpy()
    with np.errstate(invalid="ignore", over="ignore"):
        ref = np.stack([Ev[0, a == q].astype(np.float64).mean(axis=0) for q in range(keep)])
    got = merged[0].cpu().numpy().astype(np.float64)
    assert np.array_equal(np.isnan(ref), np.isnan(got))
    fin = np.isfinite(ref)
    assert np.array_equal(ref[~fin & ~np.isnan(ref)], got[~fin & ~np.isnan(ref)])
    # one unit in the last place (the sums' own rounding is 2^-24 below it)
    assert np.all(np.abs(got[fin] - ref[fin]) <= np.spacing(np.abs(ref[fin]).astype(np.float32)))


@pytest.mark.parametrize("n", [2, 3, 16, 17, 256, 257, 700, 1500])
@pytest.mark.parametrize("D", [264, 2056])
def test_fp32_means_are_correctly_rounded(n, D):
    """One centroid that gathers n rows (its group's list, ranked, and by windows): columns
    that cancel to a small part of their largest partial sum, columns spread over 2^60,
    whole numbers (ties) and subnormals. Every mean is the exact one rounded once: half a
    unit in the last place, with 2^-50 for the reference's own two roundings."""
    rng = np.random.default_rng(100 * n + D)
    Ev = rng.standard_normal((n, D)).astype(np.float32)
    first, last = rng.permutation(n)[:2]
    for c in range(D):
        k = c % 4
        if k == 0:
            big = np.float32(10.0 ** rng.uniform(4, 12))
            Ev[first, c], Ev[last, c] = big, -big
        elif k == 1:
            Ev[:, c] = np.ldexp(Ev[:, c], rng.integers(-30, 31, n))
        elif k == 2:
            Ev[:, c] = rng.integers(0, 8192, n)
        elif c < 32:
            Ev[:, c] = np.ldexp(Ev[:, c], rng.integers(-140, -120, n))
    keeps = np.array([[int(rng.integers(0, n))]], np.int32)
    _, merged = P.provip_merge(torch.from_numpy(Ev[None]).to(DEV), torch.from_numpy(keeps).to(DEV))
    torch.cuda.synchronize()
    got = merged[0, 0].cpu().numpy()
    for c in range(D):
        ref = math.fsum(Ev[:, c].astype(np.float64).tolist()) / n
        ulp = float(np.spacing(np.abs(np.float32(ref))))
        assert abs(float(got[c]) - ref) <= 0.5 * ulp + 2.0 ** -50 * abs(ref), (n, c, got[c], ref)
