"""Column-partitioned sweeps of factors whose phases or triangles take other shapes than the usual:
coarse ones, whose phases are so small that tiles have fewer entries, and sweep leaves whose
order is no multiple of eight; ops with more inputs than half a gather slice holds; and what a
NaN in one right-hand side reaches.

Bounds: a schedule with complex-FP32 coefficients, executed by the kernel's input rule, and the
device's sweeps reproduce the packed program's own sweep to 1e-5 relative (the storage rounding
and sums of a few hundred FP32 terms, as for the other sweep tests).
"""
import functools
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1901_11371_gb300", "csrc")
# factors whose lowest butterflies have rank 5 or 6: tiles of three entry pairs
RANK6 = [("arc", 1152, 72, 1e-3), ("arc", 1200, 75, 1e-2), ("strip", 1024, 128, 1e-2), ("arc", 1536, 96, 1e-2),
         ("arc", 2048, 64, 1e-1)]


@pytest.fixture(scope="session")
def sweepcheck(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path_factory.mktemp("sweepcheck") / "sweepcheck")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-fopenmp", "-I", CSRC, os.path.join(ROOT, "tests", "sweepcheck.cpp"),
                        os.path.join(CSRC, "hb_host.cpp"), os.path.join(CSRC, "hb_swsched.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]

    def run(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stdout[-2000:]
        return r.stdout.split()
    return run


@functools.lru_cache(maxsize=None)
def _hb():
    from paper_1901_11371_gb300 import build
    build.build()
    import paper_1901_11371_gb300 as m
    return m


@pytest.fixture
def hb_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return _hb()


def _geom(hb, curve, n):
    if curve == "strips8":
        return hb.hb_geometry(hb.HB_PARALLEL_STRIPS, (8.0, n / 20.0 / 8.0, 0.3), n)
    if curve == "strip":
        return hb.hb_geometry(hb.HB_STRIP, (0.0, 0.0, n / 20.0, 0.0), n)
    return hb.hb_geometry(hb.HB_ARC, (n / 20.0 / math.pi, 0.0, math.pi), n)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _check_sweeps(hb, curve, n, leaf, eps, options=0):
    """All four sweeps on the device, with one column a CTA (1, 3) and with two (155)."""
    import torch
    g = _geom(hb, curve, n)
    fh = hb.hb_factor_host(g, leaf, eps)
    f = hb.hb_factor(g, leaf, eps, form=hb.HB_C64, options=options)
    hb.hb_set_sweep_kernel(f, 1)
    for R in (1, 3, 155):
        b = W.complex_gaussian(n, 71 + R, R).T.copy()
        bt = torch.from_numpy(b[0] if R == 1 else b).cuda().to(torch.complex64)
        for w, (fn, op) in enumerate([(hb.hb_lower_solve, 0), (hb.hb_upper_solve, 0), (hb.hb_lower_solve, 1),
                                      (hb.hb_upper_solve, 1)]):
            x = fn(f, bt, op).cpu().numpy().astype(np.complex128).reshape(R, n)
            for r in {0, R // 2, R - 1}:
                assert _rel(x[r], hb.hb_host_sweep(fh, b[r], w)) <= 1e-5, (R, w, r)


@pytest.mark.parametrize("curve,n,leaf,eps", RANK6)
def test_tiles_of_three_pairs_by_the_kernels_rule(sweepcheck, curve, n, leaf, eps):
    # (such tiles must be there, with a third pair that counts)
    assert int(sweepcheck("tiles3", curve, n, leaf, eps)[1]) > 0


@pytest.mark.gpu
@pytest.mark.parametrize("curve,n,leaf,eps", RANK6)
def test_tiles_of_three_pairs_on_the_device(hb_gpu, curve, n, leaf, eps):
    _check_sweeps(hb_gpu, curve, n, leaf, eps)


def test_triangles_read_their_own_columns(sweepcheck):
    sweepcheck("triangle")


# sweep leaves of 68, 100, 84, 108 and 100 rows
@pytest.mark.gpu
@pytest.mark.parametrize("n,leaf", [(1088, 34), (1600, 50), (1344, 42), (1728, 54), (1600, 100)])
def test_sweep_leaves_off_a_multiple_of_eight_on_the_device(hb_gpu, n, leaf):
    _check_sweeps(hb_gpu, "arc", n, leaf, 1e-6)


# (factors with global phases before resident runs; tiles whose lanes read past their op's inputs)
@pytest.mark.parametrize("check,n,leaf", [("nan", 16384, 64), ("nan_small", 1600, 25), ("nan_small", 1600, 50),
                                          ("nan", 1600, 50), ("nan", 2400, 75), ("nan_small", 2400, 75)])
def test_nan_stays_in_its_column_by_the_kernels_rule(sweepcheck, check, n, leaf):
    sweepcheck(check, "arc", n, leaf, 1e-6)


@pytest.mark.gpu
@pytest.mark.parametrize("n,leaf,row,small", [(16384, 64, 8192, False), (1600, 25, 5, True), (1600, 50, 5, True)])
def test_nan_stays_in_its_column_on_the_device(hb_gpu, n, leaf, row, small):
    # 160 columns, two a CTA.  The other columns see the same sums in the same order: equal.
    import torch
    hb = hb_gpu
    f = hb.hb_factor(_geom(hb, "arc", n), leaf, 1e-6, form=hb.HB_C64, options=hb.HB_OPT_SWEEP_WINDOW_MIN if small else 0)
    hb.hb_set_sweep_kernel(f, 1)
    R, q = 160, 7
    b = torch.from_numpy(W.complex_gaussian(n, 90, R).T.copy()).cuda().to(torch.complex64)
    bad = b.clone()
    bad[q, row] = complex(float("nan"), 0.0)
    others = [r for r in range(R) if r != q]
    for fn, op in [(hb.hb_lower_solve, 0), (hb.hb_upper_solve, 0), (hb.hb_lower_solve, 1), (hb.hb_upper_solve, 1)]:
        clean, x = fn(f, b, op), fn(f, bad, op)
        assert torch.equal(x[others], clean[others])
        assert torch.isnan(torch.view_as_real(x[q, row])).any()


@pytest.mark.gpu
@pytest.mark.parametrize("small", [False, True])
@pytest.mark.parametrize("n,leaf,row", [(1600, 25, 703), (1600, 50, 405), (2400, 75, 80), (1024, 64, 129), (4096, 64, 5)])
def test_rows_that_do_not_depend_on_it_keep_their_values(hb_gpu, n, leaf, row, small):
    # A NaN, and a value whose products overflow: rows before it (L~^{-1}, U~^{-H}) or after it
    # (U~^{-1}, L~^{-H}) have the same sums in the same order: equal.
    import torch
    hb = hb_gpu
    f = hb.hb_factor(_geom(hb, "arc", n), leaf, 1e-6, form=hb.HB_C64, options=hb.HB_OPT_SWEEP_WINDOW_MIN if small else 0)
    hb.hb_set_sweep_kernel(f, 1)
    for R in (3, 160):
        b = torch.from_numpy(W.complex_gaussian(n, 90, R).T.copy()).cuda().to(torch.complex64)
        for fn, op, before in [(hb.hb_lower_solve, 0, True), (hb.hb_upper_solve, 0, False), (hb.hb_lower_solve, 1, False),
                               (hb.hb_upper_solve, 1, True)]:
            clean = fn(f, b, op)
            for value in (float("nan"), 3e38):
                bad = b.clone()
                bad[1, row] = complex(value, 0.0)
                x = fn(f, bad, op)
                free = slice(0, row) if before else slice(row + 1, n)
                assert torch.equal(x[1, free], clean[1, free]), (R, op, before, value)
                others = [r for r in range(R) if r != 1]
                assert torch.equal(x[others], clean[others]), (R, op, before, value)


# eight close strips, with global phases whose ops have 206 to 256 inputs; 400 (cut by rows; the
# scatter ops of the other two sweeps have rows of more than 384)
@pytest.mark.parametrize("n,leaf,eps,least,sweeps", [(2048, 32, 1e-6, 193, 4), (2048, 64, 1e-6, 193, 4),
                                                     (4096, 32, 1e-9, 193, 4), (4096, 64, 1e-6, 385, 2)])
def test_ops_with_many_inputs_have_a_schedule(sweepcheck, n, leaf, eps, least, sweeps):
    _, longest, _, inputs, _, built = sweepcheck("wide", "strips8", n, leaf, eps)
    assert int(longest) > 192 and int(inputs) >= least and int(built) == sweeps
    if sweeps == 4:
        sweepcheck("nan_small", "strips8", n, leaf, eps)


@pytest.mark.gpu
@pytest.mark.parametrize("n,leaf,eps", [(2048, 32, 1e-6), (2048, 64, 1e-6), (4096, 32, 1e-9)])
def test_ops_with_many_inputs_on_the_device(hb_gpu, n, leaf, eps):
    _check_sweeps(hb_gpu, "strips8", n, leaf, eps, options=hb_gpu.HB_OPT_SWEEP_WINDOW_MIN)


def test_inputs_beyond_a_runs_slots_are_refused(sweepcheck):
    sweepcheck("region", "strip", 1024, 64, 1e-6)
