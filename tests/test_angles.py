"""cos and sin of the multiples of an angle: the fixed-point table's stated error on the CPU, and on the GPU
Zernike functions next to the axes, where these are small, relative to themselves."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import trig
from paper_2409_19156_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_19156_gb300", "csrc")


def test_table_against_oracle(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe, m_max = str(tmp_path / "check"), 256
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "angle_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    axes = [q * np.pi / 2 + d for q in (-1, 0, 1, 2, 3, 4, 100) for d in (0.0, 1e-9, -1e-4, 1.9e-3)]
    off = list(np.random.default_rng(0).uniform(-2000.0, 2000.0, 12)) + [q * np.pi / 2 + 2.1e-3 for q in (0, 1, 2, 3)]
    text = "".join(f"{float(t).hex()}\n" for t in axes + off)
    lines = [[int(x) for x in line.split()] for line in subprocess.run(
        [exe, str(m_max)], input=text, capture_output=True, text=True, check=True).stdout.splitlines()]
    assert [line[0] for line in lines] == [0] * len(axes) + [1] * len(off)
    for t, line in zip(axes + off, lines):
        for m in (1, 2, 3, 16, 17, 32, 100, 128, 255, 256):
            for got, want in zip(line[2 * m - 1:2 * m + 1], trig.cos_sin_multiple(m, t)):
                assert abs(got - (want >> (trig.WORK_BITS - 62))) <= (m + 1) * 10


@pytest.mark.gpu
def test_functions_next_to_the_axes():
    """Enough points for the tables of the column walk (k = 0) and for the triangle walk (k = 1)."""
    torch, P = pytest.importorskip("torch"), 20_001
    import paper_2409_19156_gb300 as zp

    ns, ms = (np.asarray(x) for x in inputs.full_zernike_modes(15))
    base = np.array([q * np.pi / 2 + d for q in range(5) for d in (0.0, 1e-15, 1e-9, -1e-5, 1e-3)])
    which = np.arange(P) % len(base)
    r, th = (torch.as_tensor(x, device="cuda") for x in (np.ones(P), base[which]))  # R = 1 for every mode
    for k in (0, 1):
        got = zp.basis(ns, ms, r, th, k)[0][0].cpu().numpy()
        for j in np.nonzero(np.abs(ms) == ns)[0]:
            m = int(ms[j])
            want = np.array([(trig.cos_multiple(m, t) if m >= 0 else trig.sin_multiple(-m, t)) for t in base])[which]
            # m theta is next to an axis too: cos and sin are near +-1 or near m times the distance, with one
            # sign in every sum.  Angle addition rounds each factor twice per step, R twice per value.
            assert (np.abs(got[j] - want) <= 8 * (abs(m) + 1) * 2.0 ** -53 * np.abs(want)).all(), (k, m)
