"""Points that are not finite, or so far off the disc that values overflow: their own outputs alone are
affected, the same whichever form of the walk takes them, and constants stay constants."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu
BAD = [float("nan"), float("inf"), -float("inf"), 1e200]


@pytest.mark.parametrize("n_max,k", [(0, 0), (1, 2), (9, 3), (33, 1), (100, 3)])
def test_walk_forms_agree_on_bad_radii(n_max, k):
    ns, ms = inputs.radial_modes(n_max)
    plan, few = zp.Plan(ns, ms), 45
    r = torch.linspace(0.0, 1.0, few, dtype=torch.float64, device="cuda")
    r[7:11] = torch.tensor(BAD, dtype=torch.float64)
    small = zp.radial(None, None, r, k, plan=plan)  # by columns
    many = torch.rand(60_001, dtype=torch.float64, device="cuda")
    many[100:100 + few] = r     # whole waves: the triangle forms
    many[-few:] = r             # the rest
    large = zp.radial(None, None, many, k, plan=plan)
    keep = torch.ones(60_001, dtype=torch.bool, device="cuda")
    for part in (slice(100, 100 + few), slice(60_001 - few, 60_001)):
        keep[part] = False
        # (Derivatives that are constants come out as such or, by columns, as 0 * NaN.)
        assert torch.equal(torch.isfinite(large[0, :, part]), torch.isfinite(small[0]))
    assert bool((large[0, 0] == 1.0).all())  # R_0^0
    assert bool(torch.isfinite(large[:, :, keep]).all())


@pytest.mark.parametrize("n_max", [0, 1, 3, 9, 33])
def test_fused_series_of_bad_points(n_max):
    ns, ms = inputs.full_zernike_modes(n_max)
    r, th = (torch.as_tensor(x, device="cuda") for x in inputs.uniform_points(200, 2))
    r[40:43] = torch.tensor(BAD[:3], dtype=torch.float64)
    th[150] = float("nan")
    C = torch.as_tensor(inputs.scaled_normal_coeffs(ns, 3, 1), device="cuda")
    plan = zp.Plan(ns, ms)
    outs = [zp.series_eval(None, None, r, th, C, plan=plan)]
    outs += [x[:, None] for x in zp.series_adjoint(None, None, r, th, C, torch.ones((200, 3), dtype=torch.float64, device="cuda"),
                                                   need=(False, True, True), plan=plan)[1:]]
    for out in outs:
        nan = torch.isnan(out).all(1).nonzero().flatten().tolist()
        assert nan == [40, 41, 42] + ([150] if n_max else [])
        assert int(torch.isfinite(out).all(1).sum()) == 200 - len(nan)


def test_lists_without_angles_take_any_theta():
    r, _ = (torch.as_tensor(x, device="cuda") for x in inputs.uniform_points(70, 3))
    th = torch.full_like(r, float("inf"))
    C = torch.tensor([[2.0], [-1.0]], dtype=torch.float64, device="cuda")
    out = zp.series_eval([0, 2], [0, 0], r, th, C).flatten()
    # 2 - (2 r^2 - 1), the rounding of the two terms and of the sum.
    assert torch.allclose(out, 3.0 - 2.0 * r * r, rtol=0.0, atol=2.0 ** -50)
    _, gr, gt = zp.series_adjoint([0, 2], [0, 0], r, th, C, torch.ones((70, 1), dtype=torch.float64, device="cuda"))
    assert torch.allclose(gr, -4.0 * r, rtol=0.0, atol=2.0 ** -49) and bool((gt == 0.0).all())


def test_batch_with_a_list_without_angles():
    """Beside full sets, with any theta: the same bits as alone."""
    recs = []
    for ns, ms, P in (([0, 2], [0, 0], 150), (*inputs.full_zernike_modes(11), 300), ([0], [0], 40)):
        r, th = (torch.as_tensor(x, device="cuda") for x in inputs.uniform_points(P, P))
        if max(np.abs(ms)) == 0:
            th[::3] = float("nan")
        C = torch.as_tensor(np.random.default_rng(P).standard_normal((len(ns), 2)), device="cuda")
        recs.append({"n": ns, "m": ms, "r": r, "theta": th, "coeffs": C, "grad_out": torch.ones((P, 2), dtype=torch.float64, device="cuda")})
    batch = zp.Batch(recs, 2)
    batch.forward()
    batch.adjoint()
    for d, b in zip(recs, batch.instances):
        args = (d["n"], d["m"], d["r"], d["theta"], d["coeffs"])
        assert torch.equal(b["out"], zp.series_eval(*args)) and bool(torch.isfinite(b["out"]).all())
        for got, want in zip((b["grad_r"], b["grad_theta"]), zp.series_adjoint(*args, d["grad_out"], need=(False, True, True))[1:]):
            assert torch.equal(got, want) and bool(torch.isfinite(got).all())
