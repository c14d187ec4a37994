"""Where the critical text rows come first on the stream of the pre-LLM pass (host logic
compiled from the library's source, on the CPU): only where that was measured to be the
faster of the two routes."""
import os
import subprocess

import pytest

from test_merge_plan import HERE, _nvcc

# (B, N_v, N_t, D), whether they lead on 152 SMs
ROUTES = [
    # their CTAs are under three quarters of the SMs
    ((8, 2880, 96, 4096), 0), ((1, 9216, 64, 3584), 0), ((14, 576, 64, 4096), 0), ((24, 576, 64, 4096), 0),
    # a relevance CTA fits beside one of them and there is one for nearly every SM
    ((15, 576, 32, 4096), 0), ((16, 576, 64, 4096), 0), ((16, 576, 64, 2048), 0), ((29, 300, 64, 4096), 0),
    ((38, 300, 32, 4096), 0),
    # there are fewer
    ((19, 576, 32, 4096), 1), ((17, 576, 32, 5120), 1), ((32, 300, 32, 4096), 1), ((15, 300, 64, 4096), 1),
    # it does not fit, or two of them share an SM anyway
    ((16, 576, 128, 4096), 1), ((17, 576, 64, 4096), 1), ((29, 576, 32, 4096), 1), ((38, 300, 64, 4096), 1),
    ((32, 576, 64, 5120), 1), ((16, 1440, 64, 4096), 1), ((19, 1000, 32, 1024), 1),
    # the relevance has more tiles than run at once
    ((29, 1440, 64, 4096), 0), ((32, 1440, 128, 4096), 0), ((64, 576, 64, 4096), 0),
    # texts past one block are two kernels
    ((16, 576, 129, 4096), 0),
]


def test_the_critical_rows_lead_where_that_is_faster(tmp_path):
    cc = _nvcc()
    if cc is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path / "crit_route_check")
    r = subprocess.run([cc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + os.path.join(os.path.dirname(HERE), "include"),
                        os.path.join(HERE, "crit_route_check.cu"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([out, *(str(v) for s, _ in ROUTES for v in (*s, 152))], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    got = [int(x) for x in r.stdout.split()]
    assert got == [want for _, want in ROUTES], [s for (s, want), g in zip(ROUTES, got) if want != g]
