"""The work whose speed this library is judged by: its public calls at the sizes they are used at.

`listed()` names twelve cases, `draw()` gives more of the same ranges, `prepare()` makes what a
program holds before the call (points, coefficients, a plan or a batch), `run()` makes one pass
through the public entry points, `work()` counts what a pass cannot do without and `exact()`
gives the same outputs from plain torch in double-double arithmetic, rounded to float64.

The kinds of work:
  radial   radial polynomials and their rho-derivatives (tables for quadrature and fitting codes)
  basis    Zernike functions with derivatives in r and theta (design matrices, surface normals)
  series   values of Zernike series, float64-accurate or in split precision (float32 results)
  grad     one differentiable step: series values, then gradients for coefficients and points
  fit      weighted least-squares coefficients of sampled surfaces
  batch    many uneven series at once: values and all gradients (or float32 values alone)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2409_19156_gb300 as zp
from paper_2409_19156_gb300 import inputs

DEVICE = "cuda"
TWO_PI = 2.0 * math.pi


def listed() -> list[dict]:
    return [
        # The smallest call: a short radial table on a linear grid (the paper's Fig. 3 sizes), as
        # an interactive program or a set-up loop makes it thousands of times.
        {"name": "radial_n20_p100", "kind": "radial", "n_max": 20, "points": 100, "max_deriv": 0},
        # The full set of a wavefront code (231 modes) with first and second derivatives at a
        # thousand points, through the call without a plan.
        {"name": "basis_n20_p1000", "kind": "basis", "n_max": 20, "points": 1000, "max_deriv": 2, "dtheta": True,
         "plan": False},
        # One wavefront: a single coefficient set on a small aperture grid.
        {"name": "series_n20_p1000_s1", "kind": "series", "n_max": 20, "points": 1000, "sets": 1, "prec": "fp64emu"},
        # A design matrix with its gradients on an odd number of points (interferogram pixels).
        {"name": "basis_n32_p99991", "kind": "basis", "n_max": 32, "points": 99_991, "max_deriv": 1, "dtheta": True,
         "plan": True},
        # The paper's high-order table: every radial mode up to n = 100, all derivative orders.
        {"name": "radial_n100_p100000", "kind": "radial", "n_max": 100, "points": 100_000, "max_deriv": 3},
        # A few surfaces on a million points, float64-accurate.
        {"name": "series_n32_p1000000_s16", "kind": "series", "n_max": 32, "points": 1_000_000, "sets": 16,
         "prec": "fp64emu"},
        # Thousands of surfaces in float32 accuracy: the split-precision contraction.
        {"name": "series_n32_p200000_s4096_bf16x3", "kind": "series", "n_max": 32, "points": 200_000, "sets": 4096,
         "prec": "bf16x3"},
        # The other split precision, at ragged sizes.
        {"name": "series_n27_p150001_s1000_tf32", "kind": "series", "n_max": 27, "points": 150_001, "sets": 1000,
         "prec": "tf32"},
        # One optimisation step of many surfaces on a polar grid, through autograd.
        {"name": "grad_n24_p50000_s256", "kind": "grad", "n_max": 24, "points": 50_000, "sets": 256},
        # One optimisation step of a few surfaces on many scattered points.
        {"name": "grad_n32_p300007_s16", "kind": "grad", "n_max": 32, "points": 300_007, "sets": 16},
        # Coefficients of sampled surfaces, weighted.
        {"name": "fit_n24_p50000_s256", "kind": "fit", "n_max": 24, "points": 50_000, "sets": 256},
        # Uneven series of many sizes in one batch, values and gradients.
        {"name": "batch_16", "kind": "batch", "instances": 16, "n_lo": 8, "n_hi": 64, "p_lo": 1000, "p_hi": 200_000,
         "sets": 16, "prec": "fp64emu"},
    ]


def _log_int(rng, lo: float, hi: float) -> int:
    return max(1, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng) -> dict:
    kind = rng.choice(["radial", "basis", "series", "series", "grad", "grad", "fit", "batch"])
    if kind == "radial":
        n, k = _log_int(rng, 10, 100), rng.randrange(4)
        most = 1.0e9 / (_n_radial(n) * (k + 1))
        return {"kind": kind, "n_max": n, "points": _log_int(rng, 100, min(1e6, most)), "max_deriv": k}
    if kind == "basis":
        n, k = rng.randint(8, 32), rng.randrange(3)
        return {"kind": kind, "n_max": n, "points": _log_int(rng, 100, 2e5), "max_deriv": k,
                "dtheta": rng.random() < 0.5, "plan": rng.random() < 0.5}
    if kind == "series":
        n, prec = rng.randint(6, 40), rng.choice(["fp64emu", "fp64emu", "bf16x3", "tf32"])
        sets = _log_int(rng, 1, 64) if prec == "fp64emu" else _log_int(rng, 16, 4096)
        most = min(1e6, 4.5e11 / (_n_full(n) * sets), 8e8 / sets)
        if prec == "fp64emu" and sets > 16:
            most = min(most, 2e5)
        return {"kind": kind, "n_max": n, "points": _log_int(rng, 1000, max(2000, most)), "sets": sets, "prec": prec}
    if kind == "grad":
        n = rng.randint(6, 32)
        sets = _log_int(rng, 1, 256)
        return {"kind": kind, "n_max": n, "points": _log_int(rng, 1000, 3e5 if sets <= 16 else 6e4), "sets": sets}
    if kind == "fit":
        n = rng.randint(6, 24)
        return {"kind": kind, "n_max": n, "points": _log_int(rng, 20 * _n_full(n), 6e4), "sets": _log_int(rng, 1, 256)}
    lo, hi = rng.randint(6, 12), rng.randint(20, 64)
    return {"kind": kind, "instances": rng.randint(4, 16), "n_lo": lo, "n_hi": hi, "p_lo": 1000,
            "p_hi": _log_int(rng, 2e4, 2e5), "sets": rng.randint(1, 16), "prec": rng.choice(["fp64emu", "fp64emu", "fp32"])}


def _n_radial(n_max: int) -> int:
    return len(inputs.radial_modes(n_max)[0])


def _n_full(n_max: int) -> int:
    return (n_max + 1) * (n_max + 2) // 2


def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _f64(*shape, g, normal=False) -> torch.Tensor:
    f = torch.randn if normal else torch.rand
    return f(*shape, dtype=torch.float64, device=DEVICE, generator=g)


def _coeffs(n, sets: int, g) -> torch.Tensor:
    """c_nm ~ N(0, 1 / (n + 1)^2): the falling spectrum of a smooth surface."""
    scale = torch.as_tensor(1.0 / (np.asarray(n, dtype=np.float64) + 1.0), device=DEVICE)
    return _f64(len(n), sets, g=g, normal=True) * scale[:, None]


def _grid(points: int, g) -> tuple[torch.Tensor, torch.Tensor, torch.Tensor]:
    """A polar grid of `points` points (Gauss-Legendre in r^2, uniform in theta from a random
    start) and its quadrature weights; a last, part-filled ring is kept as it falls."""
    n_theta = max(8, int(round(math.sqrt(0.8 * points))))
    n_r = (points + n_theta - 1) // n_theta
    t, w = np.polynomial.legendre.leggauss(n_r)
    start = float(torch.rand((), generator=g, device=DEVICE))
    r = np.repeat(np.sqrt(0.5 * (1.0 + t)), n_theta)[:points]
    th = (np.tile(np.arange(n_theta) / n_theta, n_r)[:points] + start) % 1.0 * TWO_PI
    wt = np.repeat(w, n_theta)[:points] * (math.pi / 2 / n_theta)
    return tuple(torch.as_tensor(x, device=DEVICE) for x in (r, th, wt))


def _modes(case: dict):
    return inputs.radial_modes(case["n_max"]) if case["kind"] == "radial" else inputs.full_zernike_modes(case["n_max"])


def _batch_sizes(case: dict, seed: int) -> list[tuple[int, int]]:
    """(n_max, points) of every instance: the same for a case whatever the seed of its values."""
    rng = np.random.default_rng([case["instances"], case["n_lo"], case["n_hi"], case["p_hi"]])
    lo, hi = math.log(case["p_lo"]), math.log(case["p_hi"])
    return [(int(rng.integers(case["n_lo"], case["n_hi"] + 1)), int(round(math.exp(rng.uniform(lo, hi)))))
            for _ in range(case["instances"])]


def _values(case: dict, seed: int) -> dict:
    """The inputs of a case: tensors on the GPU, made from the seed alone."""
    g = _generator(seed)
    kind, P = case["kind"], case.get("points")
    if kind == "radial":
        # Chebyshev-distributed nodes on [0, 1], in order.
        phi = torch.sort(_f64(P, g=g), descending=True).values * math.pi
        return {"r": 0.5 * (1.0 + torch.cos(phi))}
    if kind == "basis":
        return {"r": _f64(P, g=g), "theta": _f64(P, g=g) * TWO_PI}
    n, _ = _modes(case) if kind != "batch" else (None, None)
    if kind == "series":
        return {"r": _f64(P, g=g).sqrt(), "theta": _f64(P, g=g) * TWO_PI, "coeffs": _coeffs(n, case["sets"], g)}
    if kind == "grad":
        if case["sets"] > 16:
            r, th, _ = _grid(P, g)
        else:
            r, th = _f64(P, g=g).sqrt(), _f64(P, g=g) * TWO_PI
        return {"r": r, "theta": th, "coeffs": _coeffs(n, case["sets"], g),
                "grad_out": _f64(P, case["sets"], g=g, normal=True)}
    if kind == "fit":
        r, th, w = _grid(P, g)
        x, y = r * torch.cos(th), r * torch.sin(th)
        a = _f64(6, case["sets"], g=g, normal=True)
        smooth = torch.stack([x, y, x * x - y * y, x * y, torch.sin(3.0 * x), torch.cos(2.0 * y)], 1)
        return {"r": r, "theta": th, "weights": w, "samples": smooth @ a + 0.01 * _f64(P, case["sets"], g=g, normal=True)}
    found = []
    for n_max, p in _batch_sizes(case, seed):
        nn, mm = inputs.full_zernike_modes(n_max)
        found.append({"n": nn, "m": mm, "r": _f64(p, g=g), "theta": _f64(p, g=g) * TWO_PI,
                      "coeffs": _f64(len(nn), case["sets"], g=g, normal=True),
                      "grad_out": _f64(p, case["sets"], g=g, normal=True)})
    return {"instances": found}


def prepare(case: dict, seed: int) -> dict:
    state = {"case": case, **_values(case, seed)}
    if case["kind"] == "batch":
        values_only = case["prec"] == "fp32"
        state["batch"] = zp.Batch(state["instances"], case["sets"],
                                  out_dtype=torch.float32 if values_only else torch.float64,
                                  with_adjoint=not values_only)
        return state
    n, m = _modes(case)
    if case["kind"] == "grad":
        for key in ("r", "theta", "coeffs"):
            state[key].requires_grad_()
    if case.get("plan", True):
        state["plan"] = zp.Plan(n, m)
    else:
        state["n"], state["m"] = n, m
    return state


def run(state: dict):
    case = state["case"]
    kind, plan = case["kind"], state.get("plan")
    if kind == "radial":
        return zp.radial(None, None, state["r"], case["max_deriv"], plan=plan)
    if kind == "basis":
        out, dtheta = zp.basis(state.get("n"), state.get("m"), state["r"], state["theta"], case["max_deriv"],
                               dtheta=case["dtheta"], plan=plan)
        return (out, dtheta) if case["dtheta"] else out
    if kind == "series":
        return zp.series_eval(None, None, state["r"], state["theta"], state["coeffs"], prec=case["prec"], plan=plan)
    if kind == "grad":
        wanted = (state["coeffs"], state["r"], state["theta"])
        values = zp.zernike_series(state["r"], state["theta"], state["coeffs"], plan)
        grads = torch.autograd.grad(values, wanted, grad_outputs=state["grad_out"])
        return (values.detach(), *grads)
    if kind == "fit":
        return zp.series_fit(None, None, state["r"], state["theta"], state["samples"], weights=state["weights"],
                             plan=plan)
    batch = state["batch"]
    batch.forward(case["prec"])
    if case["prec"] == "fp32":
        return [d["out"] for d in batch.instances]
    batch.adjoint()
    return [[d[k] for k in ("out", "grad_coeffs", "grad_r", "grad_theta")] for d in batch.instances]


def work(case: dict) -> dict:
    """Inputs read once, outputs written once; one multiply-add for each basis value and for
    each term of a contraction."""
    if case["kind"] == "batch":
        total = {"bytes": 0, "flops": 0}
        for n_max, p in _batch_sizes(case, 0):
            J, S = _n_full(n_max), case["sets"]
            if case["prec"] == "fp32":
                total["bytes"] += 16 * p + 8 * J * S + 4 * p * S
                total["flops"] += 2 * J * p * (S + 1)
            else:
                total["bytes"] += 2 * (16 * p + 8 * J * S) + 16 * p * S + 16 * p
                total["flops"] += 2 * J * p * (4 * S + 3)
        return total
    P, kind = case["points"], case["kind"]
    J = _n_radial(case["n_max"]) if kind == "radial" else _n_full(case["n_max"])
    if kind == "radial":
        K = case["max_deriv"] + 1
        return {"bytes": 8 * P + 8 * K * J * P, "flops": 2 * K * J * P}
    if kind == "basis":
        K = case["max_deriv"] + 1 + int(case["dtheta"])
        return {"bytes": 16 * P + 8 * K * J * P, "flops": 2 * K * J * P}
    S = case["sets"]
    if kind == "series":
        return {"bytes": 16 * P + 8 * J * S + (8 if case["prec"] == "fp64emu" else 4) * P * S,
                "flops": 2 * J * P * (S + 1)}
    if kind == "grad":
        # Values, grad_C, and the two point gradients' contractions.
        return {"bytes": 2 * (16 * P + 8 * J * S) + 16 * P * S + 16 * P, "flops": 2 * J * P * (4 * S + 3)}
    # The Gram matrix (its upper half), the right-hand side, the factorisation and the solves.
    return {"bytes": 24 * P + 8 * P * S + 8 * J * S, "flops": J * J * P + 2 * J * P * (S + 1) + J ** 3 // 3 + 2 * J * J * S}


# ---------------------------------------------------------------------------------- exact values
# Double-double arithmetic on torch float64 tensors: a pair (hi, lo) of about 106 bits.

def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _split(a):
    t = a * 134217729.0
    h = t - (t - a)
    return h, a - h


def _two_prod(a, b):
    p = a * b
    ah, al = _split(a)
    bh, bl = _split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _add(x, y):
    s, e = _two_sum(x[0], y[0])
    t, f = _two_sum(x[1], y[1])
    s, e = _two_sum(s, e + t)
    return _two_sum(s, e + f)


def _neg(x):
    return (-x[0], -x[1])


def _mul(x, y):
    p, e = _two_prod(x[0], y[0])
    return _two_sum(p, e + x[0] * y[1] + x[1] * y[0])


def _scale(x, f: float):
    """x times a whole number or a power of two."""
    p, e = _two_prod(x[0], torch.full_like(x[0], f))
    return _two_sum(p, e + x[1] * f)


def _cos_sin(theta):
    """cos and sin of theta in [0, 2 pi] as pairs: Taylor's series of theta / 64, doubled six times."""
    t = (theta / 64.0, torch.zeros_like(theta))
    t2 = _mul(t, t)
    one = (torch.ones_like(theta), torch.zeros_like(theta))

    def series(first: int):
        # sum_i (-1)^i t^(2i) first! / (2i + first)!, innermost term first.
        acc = one
        for i in range(12, 0, -1):
            d = float((2 * i + first - 1) * (2 * i + first))
            prod = _mul(acc, t2)
            q = prod[0] / d
            p, e = _two_prod(q, torch.full_like(q, d))
            rest = ((prod[0] - p) - e + prod[1]) / d
            acc = _add(one, _neg(_two_sum(q, rest)))
        return acc

    c, s = series(0), _mul(t, series(1))
    for _ in range(6):
        c, s = _add(_mul(c, c), _neg(_mul(s, s))), _scale(_mul(c, s), 2.0)
    return c, s


def _levels(n_max: int, r, orders: int):
    """For n = 0..n_max: the pairs d^k R_n^m / dr^k, k = 0..orders, each [modes, points] with
    m = n % 2, n % 2 + 2, .., n.  From R_n^m = r (R_{n-1}^{|m-1|} + R_{n-1}^{m+1}) - R_{n-2}^m and
    (R_n^m)' = n (R_{n-1}^{|m-1|} + R_{n-1}^{m+1}) + (R_{n-2}^m)'."""
    zero = torch.zeros_like(r)[None]
    rr = (r[None], zero)
    before, last = None, None
    for n in range(n_max + 1):
        if n == 0:
            now = [(torch.ones_like(zero), zero)] + [(zero, zero)] * orders
        else:
            now = []
            count = n // 2 + 1
            sums = []
            for k in range(orders + 1):
                h, low = last[k]
                pad = lambda x: torch.cat([x, zero], 0)  # noqa: E731
                if n % 2:  # m = 1, 3, ..: neighbours m - 1 = 0, 2, .. and m + 1
                    a, b = (h, low), (pad(h[1:]), pad(low[1:]))
                else:      # m = 0, 2, ..: |m - 1| = 1, 1, 3, .. and m + 1 = 1, 3, ..
                    a, b = (torch.cat([h[:1], h], 0), torch.cat([low[:1], low], 0)), (pad(h), pad(low))
                sums.append(_add(tuple(x[:count] for x in a), tuple(x[:count] for x in b)))
            for k in range(orders + 1):
                old = tuple(torch.cat([x, zero.expand(count - x.shape[0], -1)], 0) for x in before[k]) if before else \
                    (torch.zeros_like(sums[0][0]),) * 2
                if k == 0:
                    now.append(_add(_mul(rr, sums[0]), _neg(old)))
                else:
                    now.append(_add(_scale(sums[k - 1], float(n)), old))
        yield n, now
        before, last = last, now


def _basis(n_max: int, r, theta, orders: int, dtheta: bool):
    """Pairs ([orders + 1][modes, points], dtheta [modes, points]) of the full set, n then m ascending."""
    c1, s1 = _cos_sin(theta)
    cos, sin = [(torch.ones_like(theta), torch.zeros_like(theta))], [(torch.zeros_like(theta),) * 2]
    for _ in range(n_max):
        c, s = cos[-1], sin[-1]
        cos.append(_add(_mul(c, c1), _neg(_mul(s, s1))))
        sin.append(_add(_mul(s, c1), _mul(c, s1)))
    rows = [[] for _ in range(orders + 1)]
    drows = []
    stack = lambda pairs, ms: tuple(torch.stack([pairs[m][i] for m in ms]) for i in range(2))  # noqa: E731
    for n, lanes in _levels(n_max, r, orders):
        ms = list(range(n % 2, n + 1, 2))
        ct, st = stack(cos, ms), stack(sin, ms)
        first = 1 if n % 2 == 0 else 0  # m = 0 has no sine
        join = lambda neg, pos: tuple(torch.cat([x[first:].flip(0), y], 0) for x, y in zip(neg, pos))  # noqa: E731
        for k in range(orders + 1):
            rows[k].append(join(_mul(lanes[k], st), _mul(lanes[k], ct)))
        if dtheta:
            md = torch.tensor(ms, dtype=torch.float64, device=r.device)[:, None].expand_as(lanes[0][0])
            rm = _mul(lanes[0], (md, torch.zeros_like(md)))
            drows.append(join(_mul(rm, ct), _neg(_mul(rm, st))))
    cat = lambda parts: tuple(torch.cat([p[i] for p in parts], 0) for i in range(2))  # noqa: E731
    return [cat(x) for x in rows], (cat(drows) if dtheta else None)


def _slices(x, dim: int, count: int = 4, bits: int = 20):
    """Pieces of at most `bits` bits of a pair (or a tensor), on a grid common to each row along `dim`."""
    hi, lo = x if isinstance(x, tuple) else (x, torch.zeros_like(x))
    big = hi.abs().amax(dim, keepdim=True).clamp_min(1e-290)
    top = torch.exp2(torch.ceil(torch.log2(big)) + 1.0)
    found = []
    for i in range(1, count + 1):
        sigma = 1.5 * top * 2.0 ** (52 - bits * i)
        part = (hi + sigma) - sigma
        found.append(part)
        hi, lo = _two_sum(hi - part, lo)
    return found


def _matmul(a, b, most: int = 4096):
    """a [M, K] times b [K, N] (pairs or tensors) as a pair: products of slices are exact in float64."""
    total = None
    K = (a[0] if isinstance(a, tuple) else a).shape[1]
    for k in range(0, K, most):
        cut = lambda x, d: tuple(y.narrow(d, k, min(most, K - k)) for y in (x if isinstance(x, tuple) else (x,)))  # noqa: E731
        one = lambda x: x if len(x) == 2 else x[0]  # noqa: E731
        sa, sb = _slices(one(cut(a, 1)), 1), _slices(one(cut(b, 0)), 0)
        for d in range(2, 6):
            for i in range(1, d):
                if i <= len(sa) and d - i <= len(sb):
                    p = sa[i - 1] @ sb[d - i - 1]
                    total = (p, torch.zeros_like(p)) if total is None else _add(total, (p, torch.zeros_like(p)))
    return total


def _t(x):
    return tuple(y.t() for y in x)


def _exact_grad(n_max, r, theta, coeffs, grad_out, chunk=32768):
    """(values, grad_C, grad_r, grad_theta) in float64."""
    F, gC, gr, gt = [], None, [], []
    for p in range(0, r.numel(), chunk):
        z, dz = _basis(n_max, r[p:p + chunk], theta[p:p + chunk], 1, True)
        G = grad_out[p:p + chunk]
        F.append(_matmul(_t(z[0]), coeffs)[0])
        part = _matmul(z[0], G)
        gC = part if gC is None else _add(gC, part)
        for dest, d in ((gr, z[1]), (gt, dz)):
            prod = _mul(_matmul(_t(d), coeffs), (G, torch.zeros_like(G)))
            acc = (torch.zeros_like(prod[0][:, 0]),) * 2
            for s in range(prod[0].shape[1]):
                acc = _add(acc, (prod[0][:, s], prod[1][:, s]))
            dest.append(acc[0])
    return torch.cat(F), gC[0], torch.cat(gr), torch.cat(gt)


def exact(case: dict, seed: int):
    v = _values(case, seed)
    kind, n_max = case["kind"], case.get("n_max")
    if kind == "radial":
        out = torch.empty((case["max_deriv"] + 1, _n_radial(n_max), case["points"]), dtype=torch.float64, device=DEVICE)
        row = 0
        for n, lanes in _levels(n_max, v["r"], case["max_deriv"]):
            for k, lane in enumerate(lanes):
                out[k, row:row + lane[0].shape[0]] = lane[0]
            row += n // 2 + 1
        return out
    if kind == "basis":
        z, dz = _basis(n_max, v["r"], v["theta"], case["max_deriv"], case["dtheta"])
        out = torch.stack([x[0] for x in z])
        return (out, dz[0]) if case["dtheta"] else out
    if kind == "series":
        P, S = case["points"], case["sets"]
        out = torch.empty((P, S), dtype=torch.float64, device=DEVICE)
        for p in range(0, P, 32768):
            z = _basis(n_max, v["r"][p:p + 32768], v["theta"][p:p + 32768], 0, False)[0][0]
            out[p:p + 32768] = _matmul(_t(z), v["coeffs"])[0] if case["prec"] == "fp64emu" else z[0].t() @ v["coeffs"]
        return out
    if kind == "grad":
        return _exact_grad(n_max, v["r"], v["theta"], v["coeffs"], v["grad_out"])
    if kind == "fit":
        z = _basis(n_max, v["r"], v["theta"], 0, False)[0][0]
        w = v["weights"][None].expand_as(z[0])
        zw = _mul(z, (w, torch.zeros_like(w)))
        gram, rhs = _matmul(zw, _t(z)), _matmul(zw, v["samples"])
        factor = torch.linalg.cholesky(gram[0])
        c = (torch.zeros_like(rhs[0]),) * 2
        for _ in range(4):  # refinement with the residual in pairs
            rest = rhs
            for part in c:
                rest = _add(rest, _neg(_matmul(gram, part)))
            step = torch.cholesky_solve(rest[0], factor)
            c = _add(c, (step, torch.zeros_like(step)))
        return c[0]
    found = []
    for (size, _), d in zip(_batch_sizes(case, seed), v["instances"]):
        if case["prec"] == "fp32":
            parts = [_basis(size, d["r"][p:p + 32768], d["theta"][p:p + 32768], 0, False)[0][0][0].t() @ d["coeffs"]
                     for p in range(0, d["r"].numel(), 32768)]
            found.append(torch.cat(parts))
        else:
            found.append(list(_exact_grad(size, d["r"], d["theta"], d["coeffs"], d["grad_out"], 65536)))
    return found
