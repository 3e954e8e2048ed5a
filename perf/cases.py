"""Performance cases of the H-IDBF-LU library.

The work a user of the library has it do, through its public entry points: the compressed
operator's apply and adjoint apply, the FP64 residual, the approximate LU inverse
U~^{-1} L~^{-1} and its adjoint, batched solves, and the gradient of a far-field loss, from one
right-hand side to blocks of 256, from the 1,024-segment strip to the 262,144-segment
semicircle, in the three storage forms.

    listed()            the fixed cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what a program holds before the call (factor handle, right-hand sides)
    run(state)          one pass through the public entry points
    work(case)          bytes and flops one pass cannot do without
    exact(case, seed)   the same outputs from the dense matrix in 64 bits

Factor construction is timed apart in this library (hb_factor_info's build_seconds) and a
factor does not depend on the right-hand sides, so a process builds each factor once.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1901_11371_gb300 as hb
from paper_1901_11371_gb300 import autograd

FORMS = {"c128": hb.HB_C128, "c64": hb.HB_C64, "split": hb.HB_SPLIT_BF16}
ETA0, GAMMA, KAPPA = 376.73, 1.781072, 2.0 * math.pi      # wavelength 1
RTOL, RESTART = 1e-6, 30                                  # hb_gmres's defaults
ITERS = 26                                                # GMRES steps of an arc solve to RTOL
# mean ID rank of the three curve families at eps 1e-6 (what the byte and flop counts assume)
RANK = {"arc": 5, "strip": 5, "strips8": 6, "spiral": 12}


def _case(name, call, curve, n, leaf, per_wavelength, form, nrhs, adjoint=False, tuned=True):
    return {"name": name, "call": call, "curve": curve, "n": n, "leaf": leaf, "per_wavelength": per_wavelength,
            "form": form, "nrhs": nrhs, "adjoint": adjoint, "tuned": tuned}


def listed():
    return [
        # the smallest call: one apply of the 51.2-wavelength strip in the plain FP64 form (a user's own Krylov loop)
        _case("apply_strip_1k_c128_r1", "apply", "strip", 1024, 32, 20, "c128", 1),
        # one operator product of a single-wave solve on the three-turn spiral
        _case("apply_spiral_64k_c64_r1", "apply", "spiral", 65536, 64, 20, "c64", 1),
        # the adjoint product of a gradient computation on eight parallel strips
        _case("adjoint_strips8_128k_c64_r1", "apply", "strips8", 131072, 64, 40, "c64", 1, adjoint=True),
        # a few incidence angles at once, with a leaf size and a column count off the powers of two
        _case("apply_arc_50k_c64_r12", "apply", "arc", 51200, 50, 20, "c64", 12),
        # the batched benchmark's operator product: 256 angles on the semicircle, leaf contractions on tensor cores
        _case("apply_arc_256k_split_r256", "apply", "arc", 262144, 64, 40, "split", 256),
        # the refinement residual of a 40-angle solve (FP64-accurate arithmetic on complex64 factors)
        _case("residual_arc_16k_c64_r40", "residual", "arc", 16384, 64, 40, "c64", 40),
        # one preconditioner solve of a single-wave iteration
        _case("precond_spiral_64k_c64_r1", "precond", "spiral", 65536, 64, 20, "c64", 1),
        # the preconditioner on an odd number of angles, leaf size 50
        _case("precond_arc_50k_c64_r21", "precond", "arc", 51200, 50, 20, "c64", 21),
        # the adjoint preconditioner of a 16-angle gradient in the plain FP64 form
        _case("precond_h_arc_16k_c128_r16", "precond", "arc", 16384, 64, 40, "c128", 16, adjoint=True),
        # the batched benchmark's preconditioner solve (the largest case): 256 angles on the semicircle
        _case("precond_arc_256k_split_r256", "precond", "arc", 262144, 64, 40, "split", 256),
        # a whole training step through autograd: solve, far-field loss at 64 angles, adjoint solve (FP64, untuned factor)
        _case("gradient_strip_1k_c128_r1", "gradient", "strip", 1024, 32, 20, "c128", 1, tuned=False),
        # a whole batched solve with its monostatic far field: 64 angles to a true residual of 1e-6
        _case("gmres_arc_8k_split_r64", "gmres", "arc", 8192, 64, 40, "split", 64),
    ]


def draw(rng):
    call = rng.choice(["apply", "apply", "apply", "precond", "precond", "precond", "residual", "gmres"])
    form = rng.choice(["c128", "c64", "c64", "split", "split"])
    curve = rng.choice(["arc", "arc", "strip"] if call == "gmres" else ["arc", "arc", "strip", "spiral"])
    leaf = rng.choice([32, 40, 50, 56, 64, 64, 64, 72, 128])
    top = 8192 if call == "gmres" else 16384 if form == "c128" else 65536
    want = math.exp(rng.uniform(math.log(1024.0), math.log(top)))
    n = leaf << max(1, int(round(math.log2(want / leaf))))
    most = 64 if call == "gmres" or form == "c128" else 256
    most = max(1, min(most, (1 << 22) // n))
    nrhs = int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    c = _case("", call, curve, n, leaf, rng.choice([20, 40]), form, max(1, nrhs),
              adjoint=call in ("apply", "precond", "residual") and rng.random() < 0.4, tuned=rng.random() < 0.75)
    del c["name"]
    return c


# ----------------------------------------------------------------------------
# geometry, right-hand sides
# ----------------------------------------------------------------------------
def _spiral_length(theta):
    return 0.5 * (theta * math.sqrt(1.0 + theta * theta) + math.asinh(theta))


def _curve(case):
    """(kind, params) of the case's scatterer, wavelength 1."""
    length = case["n"] / case["per_wavelength"]
    if case["curve"] == "arc":
        return hb.HB_ARC, (length / math.pi, 0.0, math.pi)
    if case["curve"] == "strip":
        return hb.HB_STRIP, (0.0, 0.0, length, 0.0)
    if case["curve"] == "spiral":
        a = length / (_spiral_length(8 * math.pi) - _spiral_length(2 * math.pi))
        return hb.HB_SPIRAL, (a, 2 * math.pi, 8 * math.pi)
    return hb.HB_PARALLEL_STRIPS, (8.0, length / 8.0, 2.0)


def _segments(case):
    """Segment centres (x, y) and lengths w of the case's curve, float64 on the GPU: chords between
    nodes at equal arc length."""
    n = case["n"]
    _, p = _curve(case)
    if case["curve"] == "arc":
        t = np.linspace(p[1], p[2], n + 1)
        x, y = p[0] * np.cos(t), p[0] * np.sin(t)
    elif case["curve"] == "strip":
        x, y = np.linspace(p[0], p[2], n + 1), np.linspace(p[1], p[3], n + 1)
    elif case["curve"] == "spiral":
        s0, s1 = _spiral_length(p[1]), _spiral_length(p[2])
        s = s0 + (s1 - s0) * np.arange(n + 1) / n
        t = np.sqrt(np.maximum(2.0 * s, p[1] ** 2))
        for _ in range(30):
            r = np.sqrt(1.0 + t * t)
            t = t - (0.5 * (t * r + np.arcsinh(t)) - s) / r
        x, y = p[0] * t * np.cos(t), p[0] * t * np.sin(t)
    if case["curve"] == "strips8":
        m = n // 8
        xs = np.linspace(0.0, p[1], m + 1)
        x = np.concatenate([0.5 * (xs[1:] + xs[:-1])] * 8)
        y = np.repeat(np.arange(8) * p[2], m)
        w = np.tile(xs[1:] - xs[:-1], 8)
    else:
        w = np.hypot(np.diff(x), np.diff(y))
        x, y = 0.5 * (x[1:] + x[:-1]), 0.5 * (y[1:] + y[:-1])
    return tuple(torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (x, y, w))


def _plane_waves(case, seed):
    """exp(-i k (x cos phi + y sin phi)) for seeded incidence angles, complex128 (nrhs, n)."""
    x, y, _ = _segments(case)
    phi = np.random.default_rng(seed).uniform(0.0, math.pi, case["nrhs"])
    b = torch.empty((case["nrhs"], case["n"]), dtype=torch.complex128, device="cuda")
    for r, a in enumerate(phi):
        ph = -KAPPA * (x * math.cos(a) + y * math.sin(a))
        b[r] = torch.complex(torch.cos(ph), torch.sin(ph))
    return b, np.degrees(phi)


def _gaussian(case, seed, dtype, shape=None):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(shape or (case["nrhs"], case["n"]), dtype=dtype, device="cuda", generator=g)


def _inputs(case, seed):
    """The right-hand sides of a case: Krylov-like vectors for the operator, plane waves for the solves."""
    vec = torch.complex128 if case["form"] == "c128" else torch.complex64
    d = {}
    if case["call"] == "apply":
        d["x"] = _gaussian(case, seed, vec)
    elif case["call"] == "residual":
        d["b"], _ = _plane_waves(case, seed)
        d["x"] = _gaussian(case, seed, torch.complex128)
    elif case["call"] == "precond":
        d["b"] = _plane_waves(case, seed)[0].to(vec)
    else:
        d["b"], d["phi"] = _plane_waves(case, seed)
        if case["call"] == "gradient":
            d["obs"] = 360.0 * np.arange(64) / 64
            d["target"] = _gaussian(case, seed, torch.complex128, (case["nrhs"], 64))
    if case["nrhs"] == 1 and case["call"] in ("apply", "precond"):
        d = {k: v[0] for k, v in d.items()}
    return d


@functools.lru_cache(maxsize=24)
def _factor(curve, n, leaf, per_wavelength, form):
    kind, params = _curve({"curve": curve, "n": n, "per_wavelength": per_wavelength})
    return hb.hb_factor(hb.hb_geometry(kind, params, n), leaf, 1e-6, form=FORMS[form]), {}


def prepare(case, seed):
    f, tuned_for = _factor(case["curve"], case["n"], case["leaf"], case["per_wavelength"], case["form"])
    if case["tuned"] and tuned_for.get(case["nrhs"] > 1) != case["nrhs"]:
        hb.hb_autotune(f, case["nrhs"])     # once per factor and batch size, as a program would
        tuned_for[case["nrhs"] > 1] = case["nrhs"]
    return {"case": case, "f": f, "op": hb.HB_OP_H if case["adjoint"] else hb.HB_OP_N, **_inputs(case, seed)}


def run(state):
    f, call = state["f"], state["case"]["call"]
    if call == "apply":
        return hb.hb_apply(f, state["x"], op=state["op"])
    if call == "residual":
        return hb.hb_residual(f, state["b"], state["x"], op=state["op"])
    if call == "precond":
        return hb.hb_precond_solve(f, state["b"], op=state["op"])
    if call == "gradient":
        b = state["b"].clone().requires_grad_(True)
        loss = autograd.far_field_loss(f, b, state["target"], state["obs"], rtol=RTOL, restart=RESTART)
        return loss.detach(), torch.autograd.grad(loss, b)[0]
    x, _ = hb.hb_gmres(f, state["b"], op=state["op"], rtol=RTOL, restart=RESTART, maxit=600)
    far = hb.hb_monostatic(f, x, state["phi"])
    if state["case"]["form"] == "c128":
        return x, far
    # currents solved to 1e-6 on complex64 factors are kept in complex64
    return x.to(torch.complex64), far.to(torch.complex64)


def work(case):
    """Every stored factor entry (ID blocks, middle blocks, dense leaves) once, every vector once; eight
    flops per entry and column, and for the solves per iteration one operator and one preconditioner product."""
    n, n0, r, k = case["n"], case["leaf"], case["nrhs"], RANK[case["curve"]]
    m = n // n0
    depth = int(round(math.log2(m)))
    k = min(k, n0 // 2)
    entries = m * n0 * n0 + m * sum(2 * k * (n0 - k) + (lv + 1) * k * k for lv in range(depth))
    es = 16 if case["form"] == "c128" else 8
    vec = es if case["call"] in ("apply", "precond") else 16
    nvec = 3 if case["call"] == "residual" else 2
    products = 2 * ITERS if case["call"] == "gmres" else 4 * ITERS if case["call"] == "gradient" else 1
    return {"bytes": entries * es + nvec * n * r * vec, "flops": 8.0 * entries * r * products}


# ----------------------------------------------------------------------------
# the same outputs from the dense matrix, 64 bits
# ----------------------------------------------------------------------------
class _Dense:
    """Rows of the rescaled TM EFIE matrix a A (or its conjugate transpose), assembled block by block:
    A_ij = (k eta0 w_j / 4) H0^(2)(k |r_i - r_j|), A_ii = (k eta0 w_i / 4) [1 - i (2/pi) ln(gamma k w_i / 4e)]."""

    def __init__(self, case):
        self.n, self.h = case["n"], case["adjoint"]
        self.x, self.y, self.w = _segments(case)
        d = 1.0 - 2j / math.pi * torch.log(GAMMA * KAPPA * self.w / (4.0 * math.e)).to(torch.complex128)
        self.diag = 0.25 * KAPPA * ETA0 * self.w * d
        self.scale = 1.0 / float(self.diag.abs().max())
        self.diag = self.diag * self.scale

    def block(self, r0, r1, c0, c1):
        r = KAPPA * torch.hypot(self.x[r0:r1, None] - self.x[None, c0:c1], self.y[r0:r1, None] - self.y[None, c0:c1])
        on = torch.arange(r0, r1, device="cuda")[:, None] == torch.arange(c0, c1, device="cuda")[None, :]
        if r0 < c1 and c0 < r1:
            r = torch.where(on, torch.ones_like(r), r)
        y0 = torch.special.bessel_y0(r)
        m = torch.complex(torch.special.bessel_j0(r), y0 if self.h else -y0)
        m *= (0.25 * KAPPA * ETA0 * self.scale) * (self.w[r0:r1, None] if self.h else self.w[None, c0:c1])
        if r0 < c1 and c0 < r1:
            d = self.diag[r0:r1].conj() if self.h else self.diag[r0:r1]
            m = torch.where(on, d[:, None].expand_as(m), m)
        return m

    def apply(self, x, step=2048, wide=16384):
        """x (R, n) -> (R, n)."""
        y = torch.zeros_like(x)
        for r0 in range(0, self.n, step):
            for c0 in range(0, self.n, wide):
                r1, c1 = min(self.n, r0 + step), min(self.n, c0 + wide)
                y[:, r0:r1] += x[:, c0:c1] @ self.block(r0, r1, c0, c1).T
        return y

    def triangle(self, b, lower, unit, step=2048, wide=16384):
        """Solve with the (unit) lower or upper triangle; b (R, n)."""
        x = b.clone()
        blocks = list(range(0, self.n, step))
        for r0 in blocks if lower else reversed(blocks):
            r1 = min(self.n, r0 + step)
            lo, hi = (0, r0) if lower else (r1, self.n)
            for c0 in range(lo, hi, wide):
                c1 = min(hi, c0 + wide)
                x[:, r0:r1] -= x[:, c0:c1] @ self.block(r0, r1, c0, c1).T
            t = self.block(r0, r1, r0, r1)
            x[:, r0:r1] = torch.linalg.solve_triangular(t, x[:, r0:r1].T.contiguous(), upper=not lower,
                                                        unitriangular=unit).T
        return x

    def far(self, phi_deg):
        """F (nobs, n) of the far field E = F x."""
        phi = torch.from_numpy(np.radians(np.atleast_1d(phi_deg))).cuda()
        ph = KAPPA * (torch.cos(phi)[:, None] * self.x[None, :] + torch.sin(phi)[:, None] * self.y[None, :])
        c = -(KAPPA * ETA0 / 4.0) * np.sqrt(2j / (math.pi * KAPPA))
        return complex(c) * self.w[None, :] * torch.complex(torch.cos(ph), torch.sin(ph))


def exact(case, seed):
    n, r = case["n"], case["nrhs"]
    if n * n * (1.0 / 2.5e9 + 8.0 * r / 8e11) > 14.0:
        return None     # the dense matrix takes too long to form or to apply
    d = _inputs(case, seed)
    a = _Dense(case)
    block = lambda v: v.reshape(-1, n).to(torch.complex128)  # noqa: E731
    if case["call"] == "apply":
        return a.apply(block(d["x"])).reshape(d["x"].shape)
    if case["call"] == "residual":
        return d["b"] - a.apply(d["x"])
    if case["call"] == "precond":
        # x = U~^{-1} L~^{-1} b, or L~^{-H} U~^{-H} b: L~ unit lower, U~ upper, L~ + U~ - I = a A
        return a.triangle(a.triangle(block(d["b"]), True, not case["adjoint"]), False, case["adjoint"]).reshape(d["b"].shape)
    mat = a.block(0, n, 0, n)
    x = torch.linalg.solve(mat, (a.scale * d["b"]).T).T
    if case["call"] == "gradient":
        f = a.far(d["obs"])
        e = x @ f.T - d["target"]
        g = torch.linalg.solve(mat.conj().T, (2.0 * e @ f.conj()).T).T
        return (e.abs() ** 2).sum(), a.scale * g
    # monostatic: backscatter, the far field of column r in the direction phi_r + 180 degrees
    return x, torch.stack([a.far(p + 180.0)[0] @ x[q] for q, p in enumerate(d["phi"])])
