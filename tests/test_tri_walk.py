"""The fixed-point triangle walk that feeds the fused float64-accurate series (zp_tri.h): on the CPU
its values, read back from the digits, against the exact oracle, and its contraction layout; on
the GPU the series and the point gradients at the edges of its tiles, segments and degrees
against the float64 baseline, for full and partial mode lists and mixed on- and off-disc tiles."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import basis as obasis
from paper_2409_19156_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_19156_gb300", "csrc")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("tri") / "check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "tri_walk_check.cu"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("n_max", [0, 1, 2, 3, 7, 32, 33, 64])
def test_walk_against_oracle(driver, n_max):
    # Random angles, and those whose multiples meet the axes, where cos and sin reach +-1.
    r, th = inputs.uniform_points(40, 40 + n_max)
    r[:3], th[:4], th[4:28] = [0.0, 1.0, 1e-3], [0.0, np.pi, -1900.0, 1e-12], np.arange(24) * (np.pi / 12)
    # Radii at which R_n^0 rounds to -1, where the biased words end.
    r[28:40] = [1e-4, 1e-6, 1e-8, 3e-9, 1e-9, 1e-10, 1e-12, 1e-15, 1e-18, 5e-20, 1e-30, 1e-300]
    text = "".join(f"{float(a).hex()} {float(b).hex()}\n" for a, b in zip(r, th))
    out = subprocess.run([driver, str(n_max)], input=text, capture_output=True, text=True, check=True).stdout
    got = np.array([line.split() for line in out.splitlines()], dtype=np.int64).reshape(40, -1, 3)
    ns, ms = got[0, :, 0], got[0, :, 1]
    want = np.array(obasis.basis_table(ns, ms, r, th, 0)[0][0]).T
    # Half a unit of the last digit, the oracle's own rounding, two units of 2^-61 from each of the
    # (n / 2 + 1)^2 steps (an error spreads with weights of at most 1), and the angle: 2 pi 2^-64 times
    # |m| from the turn, four units of 2^-62 per rotation.
    steps = (n_max / 2 + 1) ** 2
    tol = 2.0 ** -54 + 2.0 ** -54 + 2 * steps * 2.0 ** -61 + (n_max + 1) * (8 * 2.0 ** -64 + 4 * 2.0 ** -62)
    assert np.max(np.abs(got[:, :, 2] * 2.0 ** -53 - want)) <= tol


def _lists(n_max, which):
    ns, ms = inputs.full_zernike_modes(n_max)
    if which == "most":  # every third mode left out, order reversed
        keep = [j for j in range(len(ns)) if j % 3 != 1][::-1]
        ns, ms = ns[keep], ms[keep]
    return ns, ms


@pytest.mark.gpu
@pytest.mark.parametrize("n_max,P,S,which", [(0, 1, 1, "full"), (1, 129, 2, "full"), (2, 128, 16, "full"),
                                             (3, 127, 9, "full"), (9, 300, 8, "most"), (31, 1, 16, "full"),
                                             (33, 1000, 7, "most"), (52, 257, 16, "full"), (54, 700, 16, "full"),
                                             (63, 20000, 3, "full"), (64, 385, 16, "most"), (65, 129, 5, "full")])
def test_series_and_gradients_against_the_baseline(n_max, P, S, which):
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp
    from paper_2409_19156_gb300 import _lib

    ns, ms = _lists(n_max, which)
    r, th = inputs.sqrt_uniform_points(P, 3 + n_max)
    if P > 300:  # a tile with points off the disc and at a negative angle among the others
        r[130:140], th[141] = np.linspace(1.0, 1.05, 10), -0.5
    C = inputs.scaled_normal_coeffs(ns, S, n_max)
    G = np.random.default_rng(n_max).standard_normal((P, S))
    r, th, C, G = (torch.as_tensor(x, device="cuda") for x in (r, th, C, G))
    plan = zp.Plan(ns, ms)
    got = [zp.series_eval(None, None, r, th, C, plan=plan)]
    got += zp.series_adjoint(None, None, r, th, C, G, need=(False, True, True), plan=plan)[1:]
    torch.cuda.synchronize()
    assert _lib.load().zp_device_wait_status(1) == 0
    want = [zp.series_eval(None, None, r, th, C, prec="fp64", plan=plan)]
    want += zp.series_adjoint(None, None, r, th, C, G, need=(False, True, True), plan=plan, prec="fp64")[1:]
    # The float64 tolerance 1e-13 of the other series tests relative to the sums of magnitudes; the
    # derivatives' are bounded by the values' over the disc times n^2 (Markov), and so are the errors
    # that the baseline's own recursion makes.
    Z, Zt = zp.basis(None, None, r, th, 1, dtheta=True, plan=plan)
    n2 = torch.as_tensor(np.maximum(ns, 1).astype(float) ** 2, device="cuda")[:, None]
    bounds = [1e-13 * (1.0 + Z[0].abs().T @ C.abs())]
    for d in (Z[1], Zt):
        bounds.append(1e-13 * (G.abs() * (1.0 + (d.abs() + n2).T @ C.abs())).sum(1))
    for g, w, b in zip(got, want, bounds):
        assert bool(((g - w).abs() <= b).all()), float(((g - w).abs() / b).max())


@pytest.mark.gpu
@pytest.mark.parametrize("n_max,k,which", [(2, 3, "full"), (9, 0, "full"), (16, 2, "most"), (33, 1, "full"), (100, 3, "radial"),
                                           (101, 0, "radial")])
def test_float64_walk_against_oracle(n_max, k, which):
    """Enough points for whole waves of the triangle form and a rest for the column form; points of
    both, at the edges of blocks and waves, at the origin, the rim, a small angle and off the disc."""
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp
    from oracle import radial as oradial

    P = 40_001
    ns, ms = inputs.radial_modes(n_max) if which == "radial" else _lists(n_max, which)
    r, th = inputs.uniform_points(P, n_max)
    rows = np.array([0, 1, 31, 32, 19_455, 19_456, 38_911, 38_912, 40_000])
    r[[0, 1, 32]], th[[31, 32]] = [0.0, 1.0, 1.02], [1e-9, -2500.0]
    if which != "radial":
        th[rows] = np.clip(th[rows], -3.0, 3.0)
    rt, tt = (torch.as_tensor(x, device="cuda") for x in (r, th))
    tol = 1e-11 * np.maximum(ns, 1).astype(float)[None, :, None] ** (2 * np.arange(k + 1))[:, None, None]
    if which == "radial":
        got = zp.radial(ns, ms, rt, k)[:, :, rows].cpu().numpy()
        want = np.array(oradial.radial_table(ns, ms, r[rows], k))
    else:
        got, dt = (x[..., rows].cpu().numpy() for x in zp.basis(ns, ms, rt, tt, k, dtheta=True))
        want, wt = obasis.basis_table(ns, ms, r[rows], th[rows], k, with_dtheta=True)
        assert (np.abs(dt - np.array(wt)) <= 1e-11 * np.maximum(ns, 1)[:, None] * 1.02 ** ns[:, None]).all()
    far = np.where(r[rows] > 1.0, 8.0 ** np.minimum(n_max, 12), 1.0)  # values beyond the rim grow past 1
    assert (np.abs(got - np.array(want)) <= tol * far).all()


@pytest.mark.gpu
@pytest.mark.parametrize("n_max,k", [(68, 3), (90, 2), (103, 3), (107, 3), (108, 3), (127, 2), (128, 2)])
def test_wide_float64_walk_against_oracle(n_max, k):
    """The form that keeps two derivative lanes in tensor memory, up to the degrees where its columns or
    its shared memory end and the next form takes over, with a rest for the one-warp and column forms."""
    pytest.importorskip("torch")
    import torch

    import paper_2409_19156_gb300 as zp
    from oracle import radial as oradial

    P = 60_001
    ns, ms = inputs.radial_modes(n_max)
    r, _ = inputs.uniform_points(P, n_max)
    rows = np.array([0, 31, 128, 255, 256, 38_911, 38_912, 58_367, 58_368, 60_000])
    r[[0, 31]] = [0.0, 1.0]
    got = zp.radial(ns, ms, torch.as_tensor(r, device="cuda"), k)[:, :, rows].cpu().numpy()
    want = np.array(oradial.radial_table(ns, ms, r[rows], k))
    tol = 1e-11 * np.maximum(ns, 1).astype(float)[None, :, None] ** (2 * np.arange(k + 1))[:, None, None]
    assert (np.abs(got - want) <= tol).all()


@pytest.mark.gpu
@pytest.mark.parametrize("prec,bound", [("bf16x3", 1e-4), ("tf32", 2e-3)])
@pytest.mark.parametrize("n_max,P,S,which", [(0, 1, 1, "full"), (1, 130, 3, "full"), (7, 127, 5, "most"), (32, 700, 20, "full"),
                                             (45, 300, 257, "most"), (64, 129, 4, "full"), (70, 129, 4, "full")])
def test_split_series_against_the_baseline(n_max, P, S, which, prec, bound):
    """Split-precision series on both sides of the triangle basis's largest degree, with whole and
    part-filled blocks: the bounds of the other split tests, relative to the sums of magnitudes."""
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp

    ns, ms = _lists(n_max, which)
    r, th = inputs.sqrt_uniform_points(P, 5 + n_max)
    if P > 500:
        r[300:303], th[303] = [1.0, 1.02, 0.0], -7.0
    C = inputs.scaled_normal_coeffs(ns, S, n_max)
    r, th, C = (torch.as_tensor(x, device="cuda") for x in (r, th, C))
    plan = zp.Plan(ns, ms)
    got = zp.series_eval(None, None, r, th, C, prec=prec, plan=plan).double()
    want = zp.series_eval(None, None, r, th, C, prec="fp64", plan=plan)
    size = zp.basis(None, None, r, th, 0, plan=plan)[0][0].abs().T @ C.abs()
    assert bool(((got - want).abs() <= bound * size + 1e-6).all())
