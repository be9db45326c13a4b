"""The fit's blocked Cholesky factorisation: mode counts at the edges of its panels of 32 against a float64
solve of the normal equations, and the same bits when its blocks start one after another because
another stream holds the GPU."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(n_modes, sets):
    n_max = int(math.ceil((math.sqrt(8 * n_modes + 1) - 3) / 2))
    ns, ms = (np.asarray(x)[:n_modes] for x in inputs.full_zernike_modes(n_max))
    r, th = inputs.polar_grid(n_max + 2, 2 * n_max + 5)
    w = np.repeat(np.polynomial.legendre.leggauss(n_max + 2)[1], 2 * n_max + 5)
    Y = np.random.default_rng(n_modes).standard_normal((len(r), sets))
    return ns, ms, *(torch.as_tensor(x, device="cuda") for x in (r, th, w, Y))


@pytest.mark.parametrize("n_modes", [1, 31, 32, 33, 64, 65, 96, 325, 640, 641, 672])
def test_panel_edges(n_modes):
    ns, ms, r, th, w, Y = _problem(n_modes, 3)
    got = zp.series_fit(ns, ms, r, th, Y, weights=w)
    Z = zp.basis(ns, ms, r, th, 0)[0][0]
    want = torch.linalg.solve((Z * w) @ Z.T, (Z * w) @ Y)
    # The quadrature makes the normal matrix nearly diagonal, of condition about 2 n_max + 2 < 80; the two
    # sums over the points and the elimination round at 2^-53 of values of order one, J times.
    assert float((got - want).abs().max()) <= 80 * 2.0 ** -50 * n_modes * (1.0 + float(want.abs().max()))


@pytest.mark.parametrize("n_modes", [325, 672])
def test_same_result_beside_another_stream(n_modes):
    ns, ms, r, th, w, Y = _problem(n_modes, 40)
    plan, other = zp.Plan(ns, ms), torch.cuda.Stream()
    quiet = zp.series_fit(None, None, r, th, Y, weights=w, plan=plan)
    rn, rm = inputs.radial_modes(60)
    busy, rr = zp.Plan(rn, rm), torch.rand(50_000, dtype=torch.float64, device="cuda")
    out = torch.empty((4, len(rn), len(rr)), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for _ in range(4):
        with torch.cuda.stream(other):
            for _ in range(6):
                zp.radial(None, None, rr, 3, plan=busy, out=out)
        assert torch.equal(zp.series_fit(None, None, r, th, Y, weights=w, plan=plan), quiet)
    torch.cuda.synchronize()
