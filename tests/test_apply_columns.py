"""Applies at the edges of their column ranges: one column through the per-step kernels (close
parallel strips, whose blocks are above the persistent kernel's staging area), and column
counts around one column thread, two slots, two columns a thread and a second CTA.

Bounds: against the oracle's host apply, 1e-13 relative for complex128 (rounding of sums of a
few hundred terms) and 1e-5 for complex-FP32 arithmetic, as for the other apply tests; the
FP64-accurate residual of a complex-FP32 factor has the factor's own rounding only, 1e-6.
"""
import math

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_11371_gb300 import build
    build.build()
    import paper_1901_11371_gb300 as m
    return m


def _geometry(hb, name):
    if name == "strips":
        return hb.hb_geometry(hb.HB_PARALLEL_STRIPS, (8.0, 6.4, 0.1), 2048), 2048, 64
    n, leaf = {"arc75": (600, 75), "arc50": (1600, 50)}[name]
    wl = W.arc(n, 1, 1e-6, radius=n / 20.0 / math.pi)
    return hb.hb_geometry(wl.kind, wl.params, n), n, leaf


@pytest.mark.parametrize("name", ["strips", "arc75", "arc50"])
@pytest.mark.parametrize("form,bound", [("HB_C128", 1e-13), ("HB_C64", 1e-5)])
def test_apply(hb, name, form, bound):
    import torch
    g, n, leaf = _geometry(hb, name)
    fh = hb.hb_factor_host(g, leaf, 1e-6)
    f = hb.hb_factor(g, leaf, 1e-6, form=getattr(hb, form))
    dt = torch.complex128 if form == "HB_C128" else torch.complex64
    x = W.complex_gaussian(n, 9, 257).T.copy()
    b = W.complex_gaussian(n, 10, 257).T.copy()
    for op in (hb.HB_OP_N, hb.HB_OP_H):
        ref = {c: hb.hb_host_apply(fh, x[c], op) for c in (0, 1, 2, 7, 8, 16, 31, 62, 63, 64, 129, 255, 256)}
        for R in (1, 2, 3, 8, 9, 17, 32, 63, 64, 65, 130, 257):
            y = hb.hb_apply(f, torch.from_numpy(x[0] if R == 1 else x[:R]).cuda().to(dt), op)
            r = hb.hb_residual(f, torch.from_numpy(b[0] if R == 1 else b[:R]).cuda(),
                               torch.from_numpy(x[0] if R == 1 else x[:R]).cuda(), op)
            y = y.cpu().numpy().astype(np.complex128).reshape(R, n)
            r = r.cpu().numpy().reshape(R, n)
            for c in ref:
                if c >= R:
                    continue
                s = np.linalg.norm(ref[c])
                assert np.linalg.norm(y[c] - ref[c]) <= bound * s, (op, R, c)
                assert np.linalg.norm(r[c] - (b[c] - ref[c])) <= (1e-13 if form == "HB_C128" else 1e-6) * s, (op, R, c)
