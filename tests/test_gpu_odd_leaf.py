"""Sweeps by the cooperative kernel on sweep leaves of odd order (odd leaf sizes above 64), whose
rows do not pair up.

Bounds against the packed program's own sweep in FP64: 1e-12 relative (FP64 sums of a few hundred
terms in another order), 1e-5 for complex-FP32, as for the other sweep tests.
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


@pytest.mark.parametrize("form,n,leaf,bound", [("HB_C128", 600, 75, 1e-12), ("HB_C64", 600, 75, 1e-5),
                                               ("HB_C128", 1048, 131, 1e-12), ("HB_C128", 1016, 127, 1e-12),
                                               ("HB_C64", 1016, 127, 1e-5)])
def test_sweeps_of_odd_leaves(hb, form, n, leaf, bound):
    import torch
    wl = W.arc(n, 1, 1e-6, radius=n / 20.0 / math.pi)
    g = hb.hb_geometry(wl.kind, wl.params, n)
    fh = hb.hb_factor_host(g, leaf, 1e-6)
    f = hb.hb_factor(g, leaf, 1e-6, form=getattr(hb, form))
    dt = torch.complex128
    if form == "HB_C64":
        hb.hb_set_sweep_kernel(f, 0)
        dt = torch.complex64
    for R in (1, 3, 40):
        b = W.complex_gaussian(n, 50 + R, R).T.copy()
        bt = torch.from_numpy(b[0] if R == 1 else b).cuda().to(dt)
        for w, (fn, op) in enumerate([(hb.hb_lower_solve, 0), (hb.hb_upper_solve, 0), (hb.hb_lower_solve, 1),
                                      (hb.hb_upper_solve, 1)]):
            x = fn(f, bt, op).cpu().numpy().astype(np.complex128).reshape(R, n)
            for r in {0, R - 1}:
                want = hb.hb_host_sweep(fh, b[r], w)
                assert np.linalg.norm(x[r] - want) <= bound * np.linalg.norm(want), (R, w, r)
