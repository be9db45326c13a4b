"""Batches whose instances ask for different gradients, through the C ABI (the Python class gives every
instance all of them): what is asked for comes out as from the single-series adjoint, the gradients of
an instance without modes or points are zeros, and nothing else is written."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2409_19156_gb300 as zp  # noqa: E402
from paper_2409_19156_gb300 import _lib, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
KEYS = ("grad_coeffs", "grad_r", "grad_theta")


# Per instance: n_max (None for no modes), points, the gradients asked for.
@pytest.mark.parametrize("spec", [
    [(5, 70, ["grad_coeffs"]), (None, 40, ["grad_r", "grad_theta"])],
    [(5, 70, ["grad_coeffs"]), (8, 0, ["grad_coeffs", "grad_r"])],
    [(9, 200, ["grad_r"]), (4, 33, ["grad_theta"]), (6, 50, []), (7, 129, ["grad_coeffs"]), (None, 3, ["grad_r"])],
    [(None, 9, ["grad_theta"])],
])
@pytest.mark.parametrize("prec", [0, 4])
def test_uneven_gradient_requests(spec, prec):
    S, rng = 3, np.random.default_rng(len(spec))
    arr = (_lib.ZpInstance * len(spec))()
    kept = []
    for a, (n_max, P, wanted) in zip(arr, spec):
        ns, ms = inputs.full_zernike_modes(n_max) if n_max is not None else (np.zeros(0, np.int32),) * 2
        ns, ms = _lib.modes_i32(ns), _lib.modes_i32(ms)
        r, th = (torch.as_tensor(x, device="cuda") for x in inputs.uniform_points(P, P))
        C, G = (torch.as_tensor(rng.standard_normal((rows, S)), device="cuda") for rows in (len(ns), P))
        shapes = {"grad_coeffs": (len(ns), S), "grad_r": (P,), "grad_theta": (P,)}
        outs = {k: torch.full(shapes[k], 7.0, dtype=torch.float64, device="cuda") for k in KEYS}
        a.n, a.m, a.n_modes = _lib.i32_ptr(ns), _lib.i32_ptr(ms), len(ns)
        a.r, a.theta, a.n_points, a.coeffs, a.grad_out = r.data_ptr(), th.data_ptr(), P, C.data_ptr(), G.data_ptr()
        for k in wanted:
            setattr(a, k, outs[k].data_ptr())
        kept.append((ns, ms, r, th, C, G, outs))
    lib, handle, st = _lib.load(), ctypes.c_void_p(), torch.cuda.current_stream().cuda_stream
    _lib.call("zp_batch_create", ctypes.cast(arr, ctypes.c_void_p), len(spec), S, ctypes.byref(handle))
    try:
        _lib.call("zp_batch_adjoint_prec", handle, prec, st)
        torch.cuda.synchronize()
        assert lib.zp_device_wait_status(1) == 0
        for (n_max, P, wanted), (ns, ms, r, th, C, G, outs) in zip(spec, kept):
            want = [torch.zeros_like(outs[k]) for k in KEYS]
            if n_max is not None and P > 0:
                want = zp.series_adjoint(ns, ms, r, th, C, G)
            for k, w in zip(KEYS, want):
                if k not in wanted:
                    assert bool((outs[k] == 7.0).all())
                else:
                    # Point gradients: sums of J S terms below 9 n^2 each, errors below 2^-50 of them; grad_C: P terms.
                    # The float64 form against the default one, so twice that: 2 * 55 * 3 * 729 * 2^-50 < 3e-10.
                    assert torch.allclose(outs[k], w, rtol=0.0, atol=3e-10)
    finally:
        _lib.call("zp_batch_destroy", handle)
