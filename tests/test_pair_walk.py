"""The split-precision basis keeps its accuracy relative to each value: on the CPU its walk in pairs of
float32 against the exact oracle, on the GPU series of high orders alone near the origin and of sines at
small angles, with no absolute slack."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import radial as oradial
from paper_2409_19156_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_19156_gb300", "csrc")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("pair") / "check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(ROOT, "tests", "pair_walk_check.cu"), "-o", exe], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("n_max", [0, 1, 4, 16, 24, 33, 71])
def test_pair_walk_against_oracle(driver, n_max):
    r = np.array([0.0, 1.0, 0.9, 0.7, 0.5, 0.4, 0.2, 0.1, 0.05, 1e-3, 1.02, 1.0 / 3.0])
    text = "".join(f"{float(x).hex()}\n" for x in r)
    out = subprocess.run([driver, str(n_max)], input=text, capture_output=True, text=True, check=True).stdout
    rows = [line.split() for line in out.splitlines()]
    count = len(rows) // len(r)
    assert count == (n_max // 2 + 1) * ((n_max + 1) // 2 + 1)
    for p, x in enumerate(r):
        part = rows[p * count:(p + 1) * count]
        ns, ms = ([int(q[i]) for q in part] for i in (0, 1))
        got = np.array([float.fromhex(q[2]) for q in part])
        want = np.array(oradial.radial_table(ns, ms, np.array([x]), 0))[0][:, 0]
        # Every value takes three roundings of at most 2^-45 of its terms; what reaches a value from the
        # (n / 2 + 1)^2 below it is no larger than it (growth region) or than 1.
        tol = 3 * (np.array(ns) / 2.0 + 1) ** 2 * 2.0 ** -45
        small = np.array(ms) >= 2.0 * x * (np.array(ns) + 1)  # well inside the growth region
        size = np.where(small, np.abs(want), np.maximum(1.0, np.abs(want)))
        # Below 2^-126 2^24 the low part leaves float32's normal range.
        assert (np.abs(got - want) <= tol * size + 2.0 ** -140 * (1.0 + tol)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("prec,bound", [("bf16x3", 1e-4), ("tf32", 2e-3)])
@pytest.mark.parametrize("n_max", [16, 24, 61, 71])
def test_high_orders_near_the_origin(n_max, prec, bound):
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp

    ns, ms = (np.asarray(x) for x in inputs.full_zernike_modes(n_max))
    r = np.array([0.4, 0.3, 0.25, 0.2] * 33)
    th = np.concatenate([np.linspace(0.1, 1.4, 66), np.tile([1e-8, -1e-6, 1e-4, 1e-13, -1e-20, 0.0], 11)])
    top = np.abs(ms) == ns
    for order in (8, 16, min(n_max, 24)):
        for sine in (False, True):
            C = np.zeros((len(ns), 2))
            C[top & (ms == (-order if sine else order))] = [1.0, -3.0]
            got = zp.series_eval(None, None, *(torch.as_tensor(x, device="cuda") for x in (r, th, C)), prec=prec,
                                 plan=zp.Plan(ns, ms)).double().cpu().numpy()
            size = r ** order  # R_m^m
            want = (size * (np.sin(order * th) if sine else np.cos(order * th)))[:, None] * np.array([1.0, -3.0])
            # The angular factor's own float32 and fixed-point roundings are absolute, below 2^-45.
            assert (np.abs(got - want) <= bound * np.abs(want) + 2.0 ** -45 * size[:, None]).all()


@pytest.mark.gpu
@pytest.mark.parametrize("prec,bound", [("bf16x3", 1e-4), ("tf32", 2e-3)])
@pytest.mark.parametrize("n_max,P", [(71, 131), (72, 131), (71, 129), (72, 385)])
def test_either_side_of_the_largest_degree(n_max, P, prec, bound):
    """n = 71 is the last degree whose tile state fits (110 KB), n = 72 takes the walk by columns."""
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp

    ns, ms = inputs.full_zernike_modes(n_max)
    r, th = inputs.sqrt_uniform_points(P, n_max)
    r[5:8], th[9] = [1.0, 1.002, 0.0], -7.0
    C = inputs.scaled_normal_coeffs(ns, 5, n_max)
    r, th, C = (torch.as_tensor(x, device="cuda") for x in (r, th, C))
    plan = zp.Plan(ns, ms)
    got = zp.series_eval(None, None, r, th, C, prec=prec, plan=plan).double()
    want = zp.series_eval(None, None, r, th, C, prec="fp64", plan=plan)
    size = zp.basis(None, None, r, th, 0, plan=plan)[0][0].abs().T @ C.abs()
    assert bool(((got - want).abs() <= bound * size).all())


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
def test_constant_at_points_that_are_not_finite(prec):
    torch = pytest.importorskip("torch")
    import paper_2409_19156_gb300 as zp

    r = torch.tensor([0.5, float("nan"), float("inf"), 2.0], dtype=torch.float64, device="cuda")
    C = torch.full((1, 1), 0.75, dtype=torch.float64, device="cuda")
    assert zp.series_eval([0], [0], r, torch.zeros_like(r), C, prec=prec).flatten().tolist() == [0.75] * 4
