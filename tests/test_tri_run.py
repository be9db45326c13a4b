"""Segments of the fused series' contraction are short enough for exact float32 sums, also for points off
the disc, whose leading digits are larger: on the CPU by the layout and the digits themselves, on the GPU
at the degrees whose triangle is the longest that one segment holds and the next ones."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2409_19156_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_19156_gb300", "csrc")


def test_diagonal_sums_stay_exact(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "tri_run_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    lines = [[int(x) for x in line.split()] for line in subprocess.run([exe], capture_output=True, text=True,
                                                                       check=True).stdout.splitlines()]
    lead, digits = lines[0]
    # Values: `lead`, then 32; coefficients: at most 2^6 + 1, then 32.  Diagonal d holds a_0 b_d, a_d b_0 and
    # d - 1 products of later digits.
    most = max(lead * 65 if d == 0 else lead * 32 + 65 * 32 + (d - 1) * 32 * 32 for d in range(digits))
    for positions, held, chunks in lines[1:]:
        assert positions * most < 2 ** 24
        assert held >= chunks


@pytest.mark.gpu
@pytest.mark.parametrize("n_max", [50, 51, 52, 53, 54])
def test_off_disc_points_at_the_longest_segments(n_max):
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp

    ns, ms = inputs.full_zernike_modes(n_max)
    P, S = 257, 16
    r, th = inputs.sqrt_uniform_points(P, n_max)
    r[::3] = np.linspace(1.0 + 2.0 ** -52, 1.02, len(r[::3]))
    C = np.random.default_rng(n_max).choice([-1.0, 1.0], (len(ns), S))
    r, th, C = (torch.as_tensor(x, device="cuda") for x in (r, th, C))
    plan = zp.Plan(ns, ms)
    got = zp.series_eval(None, None, r, th, C, plan=plan)
    want = zp.series_eval(None, None, r, th, C, prec="fp64", plan=plan)
    # As for the other series: 1e-13 of the sums of magnitudes; the scale is the row's largest value.
    Z = zp.basis(None, None, r, th, 0, plan=plan)[0][0].abs()
    size = Z.T @ C.abs() + len(ns) * 2.0 ** -52 / 1e-13 * Z.max(0).values[:, None]
    assert bool(((got - want).abs() <= 1e-13 * size).all()), float(((got - want).abs() / size).max())
