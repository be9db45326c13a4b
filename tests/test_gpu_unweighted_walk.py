"""grad_coeffs of calls large enough (2^23 basis values) for the walk that leaves out the recursion
weights: its 32- and 128-thread forms, odd point counts, duplicated and sparse modes, points off the
disc and points that are not finite, against float64 sums over the basis itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _sparse(n_max, step):
    ns, ms = (np.asarray(x) for x in inputs.full_zernike_modes(n_max))
    keep = np.arange(len(ns))[::step]
    return ns[keep], ms[keep]


@pytest.mark.parametrize("name,modes,P", [
    ("many columns, few points: 32-thread blocks", inputs.full_zernike_modes(180), 513),
    ("odd points, 32-thread blocks", inputs.full_zernike_modes(100), 1637),
    ("odd points, tables, 128-thread blocks", inputs.full_zernike_modes(24), 25_825),
    ("even points, tables", inputs.full_zernike_modes(24), 25_812),
    ("sparse", _sparse(60, 7), 31_089),
    ("duplicates", tuple(np.concatenate([x, x[::3], x[:5], x[:5]]) for x in map(np.asarray, inputs.full_zernike_modes(20))), 30_001),
])
@pytest.mark.parametrize("off", [False, True])
def test_grad_coeffs_against_sums(name, modes, P, off):
    ns, ms = modes
    assert len(ns) * P >= 2 ** 23
    r, th = inputs.sqrt_uniform_points(P, 11)
    if off:
        r[[0, 1, P // 2, P - 1]] = [1.01, 1.0 + 2.0 ** -52, 1.005, 1.01]
        th[[2, 3]] = [-3.0, 7000.0]
    S = 5
    r, th = (torch.as_tensor(x, device="cuda") for x in (r, th))
    C = torch.zeros((len(ns), S), dtype=torch.float64, device="cuda")
    G = torch.as_tensor(np.random.default_rng(P).standard_normal((P, S)), device="cuda")
    plan = zp.Plan(ns, ms)
    got = zp.series_adjoint(None, None, r, th, C, G, need=(True, False, False), plan=plan)[0]
    Z = zp.basis(None, None, r, th, 0, plan=plan)[0][0]
    want = Z @ G
    # The GEMM's bound, P 2^-54 of the row's largest |Z| and the column's largest |G|; the walks' own errors, at
    # most 1e-13 of the sums of magnitudes as in the other series tests; the float64 sum's.
    bound = P * 2.0 ** -52 * Z.abs().max(1).values[:, None] * G.abs().max(0).values + 1e-13 * (Z.abs() @ G.abs())
    assert bool(((got - want).abs() <= bound).all()), (name, float(((got - want).abs() / bound).max()))


def test_a_point_that_is_not_finite_spoils_every_mode_that_sees_it():
    ns, ms = inputs.full_zernike_modes(24)
    P = 25_825
    r, th = (torch.as_tensor(x, device="cuda") for x in inputs.sqrt_uniform_points(P, 1))
    r[P - 1] = float("nan")
    G = torch.ones((P, 2), dtype=torch.float64, device="cuda")
    C = torch.zeros((len(ns), 2), dtype=torch.float64, device="cuda")
    gC = zp.series_adjoint(ns, ms, r, th, C, G, need=(True, False, False))[0]
    assert bool(torch.isnan(gC[1:]).all()) and bool(torch.isfinite(gC[0]).all())  # (0, 0) is constant
