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
    off += [2047.5, 2100.0, -5000.0, 1e6, 1e9, -3.0e12, 2.0 ** 51 + 0.5, 2.0 ** 52 - 0.5]  # large angles too
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


@pytest.mark.gpu
def test_series_at_large_angles():
    """Angles up to 2^52 against the oracle: the fused series, its gradients and the split basis."""
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp
    from oracle import basis as obasis

    ns, ms = inputs.full_zernike_modes(20)
    th = np.array([2047.0, 2048.0, -2049.0, 5000.25, 1e6, -1e9, 3.0e12, 2.0 ** 51 + 0.5, 2.0 ** 52 - 0.5, 2.0 ** 52, 1e17])
    r = np.linspace(0.1, 1.0, len(th))
    C = inputs.scaled_normal_coeffs(ns, 3, 5)
    z, zt = (np.array(x) for x in obasis.basis_table(ns, ms, r, th, 1, with_dtheta=True))
    plan, G = zp.Plan(ns, ms), np.ones((len(th), 3))
    rt, tt, Ct, Gt = (torch.as_tensor(x, device="cuda") for x in (r, th, C, G))
    F = zp.series_eval(None, None, rt, tt, Ct, plan=plan).cpu().numpy()
    size = np.abs(C).sum(0)
    assert (np.abs(F - z[0].T @ C) <= 1e-13 * (1.0 + size)).all()
    gr, gt = (x.cpu().numpy() for x in zp.series_adjoint(None, None, rt, tt, Ct, Gt, need=(False, True, True), plan=plan)[1:])
    for got, d in ((gr, z[1]), (gt, zt)):  # derivatives of up to n^2 <= 400 per mode
        assert (np.abs(got - (d.T @ C).sum(1)) <= 1e-13 * (1.0 + 400.0 * size.sum())).all()
    got = zp.series_eval(None, None, rt, tt, Ct, prec="bf16x3", plan=plan).double().cpu().numpy()
    assert (np.abs(got - z[0].T @ C) <= 1e-4 * (np.abs(z[0]).T @ np.abs(C))).all()
