"""Column-major blocks of right-hand sides through the tiled layout changes: row counts that
are no multiple of a tile, right-hand-side counts at the edges of a tile, and blocks with a
leading dimension above N.

Bounds: against the oracle's host apply, 1e-13 relative for complex128 (rounding of sums of a
few hundred terms) and 1e-5 for complex-FP32 arithmetic, as for the other apply tests; rows
of padding between the columns stay as they were.
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


@pytest.mark.parametrize("form,bound", [("HB_C128", 1e-13), ("HB_C64", 1e-5)])
@pytest.mark.parametrize("n,leaf,nrhs,pad", [(600, 75, 2, 0), (600, 75, 33, 5), (1600, 50, 31, 1), (1600, 50, 65, 0)])
def test_blocks_of_columns(hb, form, bound, n, leaf, nrhs, pad):
    import ctypes as C
    import torch
    wl = W.arc(n, 1, 1e-6, radius=n / 20.0 / math.pi)
    g = hb.hb_geometry(wl.kind, wl.params, n)
    fh = hb.hb_factor_host(g, leaf, 1e-6)
    f = hb.hb_factor(g, leaf, 1e-6, form=getattr(hb, form))
    dt = torch.complex128 if form == "HB_C128" else torch.complex64
    x = W.complex_gaussian(n, 5, nrhs).T.copy()
    b = W.complex_gaussian(n, 6, nrhs).T.copy()
    ld = n + pad

    def padded(v, dtype):
        t = torch.full((nrhs, ld), 7.0, dtype=dtype, device="cuda")
        t[:, :n] = torch.from_numpy(v).cuda().to(dtype)
        return t

    lib = hb.lib()
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    xd, y = padded(x, dt), padded(0 * x, dt)
    hb._lib.check(lib.hb_apply(f._h, hb.HB_OP_N, C.c_void_p(xd.data_ptr()), C.c_void_p(y.data_ptr()), nrhs, ld, st))
    xr, bd, r = padded(x, torch.complex128), padded(b, torch.complex128), padded(0 * x, torch.complex128)
    hb._lib.check(lib.hb_residual(f._h, hb.HB_OP_N, C.c_void_p(bd.data_ptr()), C.c_void_p(xr.data_ptr()),
                                  C.c_void_p(r.data_ptr()), nrhs, ld, st))
    ref = np.stack([hb.hb_host_apply(fh, x[c]) for c in range(nrhs)])
    for out, want in ((y, ref), (r, b - ref)):
        got = out[:, :n].cpu().numpy().astype(np.complex128)
        for c in range(nrhs):
            assert np.linalg.norm(got[c] - want[c]) <= bound * np.linalg.norm(ref[c]), c
        assert bool((out[:, n:] == 7.0).all())
