"""Column-partitioned sweeps off the usual sizes: leaf sizes whose rows do not pair up (odd),
that are no power of two, or above the 128-row sweep leaf, on the host schedule and on the GPU.

Bounds: the schedule with complex128 coefficients reproduces the packed program's own sweep to
rounding (1e-13); complex-FP32 coefficients and arithmetic give 1e-5 relative, as for the other
sweep tests.  A NaN in one row of one right-hand side must leave the other right-hand sides
bitwise as they were and, in L~^{-1} (rows in order), every earlier row finite.
"""
import math

import numpy as np
import pytest

import workloads as W

SIZES = [(1600, 25), (1600, 50), (2400, 75), (2400, 150), (1024, 8)]


@pytest.fixture(scope="module")
def hb():
    from paper_1901_11371_gb300 import build
    build.build()
    import paper_1901_11371_gb300 as m
    return m


def _geom(hb, n):
    wl = W.arc(n, 1, 1e-6, radius=n / 20.0 / math.pi)
    return hb.hb_geometry(wl.kind, wl.params, n)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,leaf", SIZES)
def test_schedule_matches_host_sweep(hb, n, leaf):
    f = hb.hb_factor_host(_geom(hb, n), leaf, 1e-6)
    b = W.complex_gaussian(n, 70)
    for which in range(4):
        ref = hb.hb_host_sweep(f, b, which)
        for win in (0, 512):
            x, _ = hb.hb_host_sweep_sched(f, b, which, 16, win_slots=win)
            assert _rel(x, ref) <= 1e-13, (which, win)
            x, _ = hb.hb_host_sweep_sched(f, b, which, 8, win_slots=win)
            assert _rel(x, ref) <= 1e-5, (which, win)


@pytest.mark.gpu
@pytest.mark.parametrize("n,leaf", SIZES)
def test_sweeps_on_the_device(hb, n, leaf):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = _geom(hb, n)
    fh = hb.hb_factor_host(g, leaf, 1e-6)
    for opts in (0, hb.HB_OPT_SWEEP_WINDOW_MIN):
        try:
            f = hb.hb_factor(g, leaf, 1e-6, form=hb.HB_C64, options=opts)
        except hb.HBError as e:
            assert e.code == hb._lib.HB_EUNSUPPORTED
            pytest.skip(f"leaf size refused by the device image: {e}")
        hb.hb_set_sweep_kernel(f, 1)
        for R in (1, 3, 155):
            b = W.complex_gaussian(n, 71 + R, R).T.copy()
            bt = torch.from_numpy(b[0] if R == 1 else b).cuda().to(torch.complex64)
            for w, (fn, op) in enumerate([(hb.hb_lower_solve, 0), (hb.hb_upper_solve, 0), (hb.hb_lower_solve, 1),
                                          (hb.hb_upper_solve, 1)]):
                x = fn(f, bt, op).cpu().numpy().astype(np.complex128).reshape(R, n)
                for r in {0, R // 2, R - 1}:
                    assert _rel(x[r], hb.hb_host_sweep(fh, b[r], w)) <= 1e-5, (opts, R, w, r)


@pytest.mark.gpu
@pytest.mark.parametrize("n,leaf,row", [(1600, 25, 777), (1024, 64, 900), (1024, 64, 129)])
def test_nan_stays_in_its_column_and_below_its_row(hb, n, leaf, row):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    f = hb.hb_factor(_geom(hb, n), leaf, 1e-6, form=hb.HB_C64)
    hb.hb_set_sweep_kernel(f, 1)
    for R in (3, 160):
        b = torch.from_numpy(W.complex_gaussian(n, 90, R).T.copy()).cuda().to(torch.complex64)
        clean = hb.hb_lower_solve(f, b)
        b[1, row] = complex(float("nan"), 0.0)
        x = hb.hb_lower_solve(f, b)
        others = [r for r in range(R) if r != 1]
        assert torch.isfinite(torch.view_as_real(x[1, :row])).all()
        assert torch.isnan(torch.view_as_real(x[1, row])).any()
        assert _rel(x[others].cpu().numpy(), clean[others].cpu().numpy()) <= 1e-5
        if R == 3:   # (one right-hand side per CTA)
            assert torch.equal(x[others], clean[others])
