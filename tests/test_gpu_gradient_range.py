"""Point gradients of at most 16 sets over the whole range of float64: coefficients scaled by a power of
two give gradients scaled by the same power, bit for bit, as far as these are normal numbers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_max", [1, 2, 3, 20, 64])
@pytest.mark.parametrize("power", [1004, 998, 900, -900])
def test_gradients_scale_with_the_coefficients(n_max, power):
    ns, ms = inputs.full_zernike_modes(n_max)
    r, th = inputs.uniform_points(77, n_max)
    # |dZ| <= n^2 and (n + 1) modes of each n: this spectrum keeps gradients below 2^(power + 8).
    C = np.sign(inputs.scaled_normal_coeffs(ns, 5, n_max)) / (np.asarray(ns)[:, None] + 1.0) ** 3
    C[:, 1] *= 2.0 ** -40  # sets of their own scale
    G = np.eye(77, 5)
    r, th, C, G = (torch.as_tensor(x, device="cuda") for x in (r, th, C, G))
    plan = zp.Plan(ns, ms)
    want = zp.series_adjoint(None, None, r, th, C, G, need=(False, True, True), plan=plan)[1:]
    got = zp.series_adjoint(None, None, r, th, C * 2.0 ** power, G, need=(False, True, True), plan=plan)[1:]
    for g, w in zip(got, want):
        assert bool(torch.isfinite(g).all())
        assert torch.equal(g * 2.0 ** -power, w)


@pytest.mark.parametrize("n_max", [20, 64])
def test_gradients_at_the_top_of_the_range(n_max):
    """One mode (n, 0) with a coefficient of 2^1020 near the origin: its Cartesian derivatives hold
    coefficients 2 (n - 1) times as large, beyond float64, its gradient n (n + 2) r / 2 times, within."""
    ns, ms = (np.asarray(x) for x in inputs.full_zernike_modes(n_max))
    r, th = np.linspace(0.0, 0.002, 50), np.linspace(0.3, 6.0, 50)
    C = np.zeros((len(ns), 1))
    C[(ns == n_max) & (ms == 0)] = 1.0
    r, th, C, G = (torch.as_tensor(x, device="cuda") for x in (r, th, C, np.ones((50, 1))))
    plan = zp.Plan(ns, ms)
    want = zp.series_adjoint(None, None, r, th, C, G, need=(False, True, False), plan=plan)[1]
    got = zp.series_adjoint(None, None, r, th, C * 2.0 ** 1020, G, need=(False, True, False), plan=plan)[1]
    assert float(want.abs().max()) < 8.0
    assert torch.equal(got * 2.0 ** -1020, want)


def test_sets_that_are_not_finite_alone_give_nan():
    ns, ms = inputs.full_zernike_modes(12)
    r, th = (torch.as_tensor(x, device="cuda") for x in inputs.uniform_points(40, 1))
    plan, G = zp.Plan(ns, ms), torch.zeros((40, 4), dtype=torch.float64, device="cuda")
    C = torch.as_tensor(inputs.scaled_normal_coeffs(ns, 4, 2), device="cuda")
    C[3, 1], C[-1, 2] = float("inf"), float("nan")
    for s in range(4):
        one = G.clone()[:, s:s + 1] + 1.0
        for g in zp.series_adjoint(None, None, r, th, C[:, s:s + 1].contiguous(), one, need=(False, True, True), plan=plan)[1:]:
            assert bool(torch.isfinite(g).all()) == (s in (0, 3))
            assert bool(torch.isnan(g).all()) == (s in (1, 2))
