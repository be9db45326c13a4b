"""Tensor-memory loads and stores are whole-warp instructions: calls whose last warp is part filled, and
warps whose points take different branches, against the float64 baseline."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import _lib, inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1, 15, 31, 33, 63, 65, 127, 129, 191, 20_001])
@pytest.mark.parametrize("S", [1, 8, 9, 16, 20])
def test_gradients_of_part_filled_warps(P, S):
    ns, ms = inputs.full_zernike_modes(13)
    r, th = inputs.sqrt_uniform_points(P, P)
    r[::7] = 0.0        # R = 0 or +-1: zero sums beside others
    r[3::11] = 1.0001   # another row scale in the same warp
    C = inputs.scaled_normal_coeffs(ns, S, P)
    C[:, -1] = 0.0
    G = np.random.default_rng(P).standard_normal((P, S))
    r, th, C, G = (torch.as_tensor(x, device="cuda") for x in (r, th, C, G))
    plan = zp.Plan(ns, ms)
    got = [zp.series_eval(None, None, r, th, C, plan=plan), *zp.series_adjoint(None, None, r, th, C, G, plan=plan)]
    torch.cuda.synchronize()
    assert _lib.load().zp_device_wait_status(1) == 0
    want = [zp.series_eval(None, None, r, th, C, prec="fp64", plan=plan),
            *zp.series_adjoint(None, None, r, th, C, G, prec="fp64", plan=plan)]
    # 1e-13 of the sums of magnitudes, as for the other series tests: |Z| <= 1.01, |dZ| <= 1.01 n^2.
    Ca, Ga, n2 = C.abs(), G.abs(), torch.as_tensor(np.maximum(ns, 1).astype(float) ** 2, device="cuda")
    sums = [Ca.sum(0).expand(P, S), Ga.sum(0).expand(len(ns), S), *[(Ga * (n2 @ Ca)).sum(1)] * 2]
    for g, w, b in zip(got, want, sums):
        assert bool(((g - w).abs() <= 1e-13 * (1.0 + 1.1 * b)).all()), float((g - w).abs().max())
