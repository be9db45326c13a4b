"""grad_theta of at most 16 sets comes from Cartesian derivatives, r (cos F_y - sin F_x): its error is measured
by the gradient's size, and stays within the functions' own bound |dZ/dtheta| <= |m| <= n."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_max", [3, 20, 32, 64])
@pytest.mark.parametrize("symmetric", [False, True])
def test_grad_theta_against_the_baseline(n_max, symmetric):
    ns, ms = (np.asarray(x) for x in inputs.full_zernike_modes(n_max))
    P, S = 1003, 7
    r, th = inputs.sqrt_uniform_points(P, n_max)
    C = inputs.scaled_normal_coeffs(ns, S, 3)
    if symmetric:
        C[ms != 0] = 0.0
    G = np.random.default_rng(1).standard_normal((P, S))
    n1 = torch.as_tensor(np.maximum(ns, 1).astype(float), device="cuda")
    r, th, C, G = (torch.as_tensor(x, device="cuda") for x in (r, th, C, G))
    plan = zp.Plan(ns, ms)
    got = zp.series_adjoint(None, None, r, th, C, G, need=(False, False, True), plan=plan)[2]
    if symmetric:
        want = torch.zeros_like(got)
    else:
        want = zp.series_adjoint(None, None, r, th, C, G, need=(False, False, True), plan=plan, prec="fp64")[2]
    # The float64 tolerance 1e-13 of the other series tests, relative to the sums with |dZ/dtheta| <= n.
    bound = 1e-13 * (G.abs() * (n1 @ C.abs())).sum(1)
    assert bool(((got - want).abs() <= bound).all()), float(((got - want).abs() / bound).max())
