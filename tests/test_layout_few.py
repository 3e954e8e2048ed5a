"""Blocks of few right-hand sides, and one, through the layout changes that go element by element,
around the counts where the tiles take over; leading dimensions above N.

Bounds: a layout change moves values without arithmetic, so with an operator applied to each
column alone and to the block the results agree to the rounding of sums in another order: 1e-13
relative (FP64), 1e-5 (complex-FP32), as for the other apply tests; padding stays as it was.
"""
import ctypes as C
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
@pytest.mark.parametrize("nrhs,pad", [(1, 0), (1, 3), (2, 1), (10, 0), (11, 5), (20, 1), (21, 0)])
def test_blocks_of_few_columns(hb, form, bound, nrhs, pad):
    import torch
    n, leaf = 600, 75
    wl = W.arc(n, 1, 1e-6, radius=n / 20.0 / math.pi)
    g = hb.hb_geometry(wl.kind, wl.params, n)
    fh = hb.hb_factor_host(g, leaf, 1e-6)
    f = hb.hb_factor(g, leaf, 1e-6, form=getattr(hb, form))
    dt = torch.complex128 if form == "HB_C128" else torch.complex64
    x = W.complex_gaussian(n, 5, nrhs).reshape(n, nrhs).T.copy()
    b = W.complex_gaussian(n, 6, nrhs).reshape(n, nrhs).T.copy()
    ld = n + pad

    def padded(v, dtype):
        t = torch.full((nrhs, ld), 7.0, dtype=dtype, device="cuda")
        t[:, :n] = torch.from_numpy(v).cuda().to(dtype)
        return t

    def call(name, *bufs):
        st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        hb._lib.check(getattr(hb.lib(), name)(f._h, hb.HB_OP_N, *[C.c_void_p(t.data_ptr()) for t in bufs], nrhs, ld, st))

    xd, y, z = padded(x, dt), padded(0 * x, dt), padded(0 * x, dt)
    xr, bd, r = padded(x, torch.complex128), padded(b, torch.complex128), padded(0 * x, torch.complex128)
    call("hb_apply", xd, y)
    call("hb_precond_solve", xd, z)
    call("hb_residual", bd, xr, r)
    ref = np.stack([hb.hb_host_apply(fh, x[c]) for c in range(nrhs)])
    pre = np.stack([hb.hb_host_sweep(fh, hb.hb_host_sweep(fh, x[c], 0), 1) for c in range(nrhs)])
    for out, want, scale in ((y, ref, ref), (z, pre, pre), (r, b - ref, ref)):
        got = out[:, :n].cpu().numpy().astype(np.complex128)
        for c in range(nrhs):
            assert np.linalg.norm(got[c] - want[c]) <= bound * np.linalg.norm(scale[c]), c
        assert bool((out[:, n:] == 7.0).all())
