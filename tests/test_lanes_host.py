"""The passes of csrc/solver.cuh with every thread of a CTA as a fiber of its own
(tests/lanes): between two barriers a whole lane runs before the next one, in
either order, and a shuffle orders no memory.  A hand-over through shared memory
without a barrier gives wrong results here; on a GPU it may or may not.

Tolerances: an FP32 line is transformed forward and back, 2 log2(n) stages of at
most 2^-23 relative each to the largest value: 18 2^-23 < 2.2e-6 for 512 points,
3e-6 with the conversions; an FP64 one 18 2^-52: 4e-15."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2204_07247_gb300", "csrc")


@pytest.fixture(scope="module")
def lanes(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("lanes"))
    for src in (CSRC, os.path.join(HERE, "lanes")):  # the latter's compat.cuh replaces the former's
        for f in os.listdir(src):
            if f.endswith((".cuh", ".cpp")):
                shutil.copy(os.path.join(src, f), d)
    so = os.path.join(d, "liblanes.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-w", "-fno-strict-aliasing", "-fPIC", "-shared", "-o", so,
                           os.path.join(d, "lanes.cpp")])
    return ctypes.CDLL(so)


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def spectrum(k, lead, rows, seed):
    """k fields of half spectra [field][lead][rows], real in the first and last of lead"""
    r = np.random.default_rng(seed)
    s = r.uniform(-1, 1, (k, lead, rows)) + 1j * r.uniform(-1, 1, (k, lead, rows))
    s[:, [0, -1]] = s[:, [0, -1]].real
    return s


PASSES = [("col_sum_fx", 3), ("col_sum_coop_fx", 3), ("row_fx", 3), ("row_coop_fx", 3), ("col_fx", 3), ("col_coop_fx", 3),
          ("row_coop", 2), ("col_coop", 2), ("mid_fx_fwd", 2), ("mid_fx_inv", 2), ("row_staged", 1), ("row_staged", 2),
          ("col_staged", 1), ("col_staged", 2), ("row_pair", 2), ("col_pair", 2), ("mid_staged_fwd", 2), ("mid_staged_inv", 2)]
# (points of a line, compile-time length or 0; the staged passes have compile-time lengths only)
CASES = [(p, k, n, nf) for p, k in PASSES for n, nf in [(8, 0), (16, 0), (32, 0), (64, 0), (128, 0), (64, 64), (128, 128), (512, 512)]
         if nf or not ("staged" in p or "pair" in p)]


@pytest.mark.parametrize("up", [1, 0])
@pytest.mark.parametrize("name,k,n,nf", CASES)
def test_passes_do_not_depend_on_the_order_of_lanes(lanes, name, k, n, nf, up):
    if name[0] == "r":      # [k][n / 2 + 1][8 rows]: inverse and forward along n, scaled by 1 / (8 n)
        src = spectrum(k, n // 2 + 1, 8, n)
        want = src / 8
    elif name[0] == "c":    # [k][5 lines][n]: forward and inverse along n
        src = spectrum(k, 5, n, n)
        want = src * n
        if "sum" in name:
            want = np.concatenate([want.sum(0, keepdims=True), np.zeros((k - 1,) + want.shape[1:])])
    else:                   # [k][5 planes][8 lines][n] <-> [k][5][n][8]
        src = spectrum(k, 5, 8 * n, n)
        if "fwd" in name:
            want = np.swapaxes(np.fft.fft(src.reshape(k, 5, 8, n)), 2, 3)
        else:
            want = n * np.fft.ifft(np.swapaxes(src.reshape(k, 5, n, 8), 2, 3))
    src = np.ascontiguousarray(src)
    dst = np.zeros_like(src)
    assert lanes.lanes_pass(name.encode(), n, nf, k, up, ctypes.c_double(0), ptr(src), ptr(dst)) == 1
    tol = 4e-15 if name.endswith("_fx") and "sum" not in name or "mid_fx" in name else 3e-6
    assert np.abs(dst - want.reshape(dst.shape)).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("n", [64, 512])
@pytest.mark.parametrize("axis", ["row", "col"])
def test_pairs_of_warps_give_the_bits_of_one(lanes, axis, n):
    """The pair passes do the arithmetic of the staged ones: the same bits, with
    pointwise state that differs from point to point and field to field."""
    src = spectrum(2, n // 2 + 1, 8, n) if axis == "row" else spectrum(2, 5, n, n)
    src, out = np.ascontiguousarray(src), []
    for form in ("staged", "pair"):
        dst = np.zeros_like(src)
        assert lanes.lanes_pass(f"{axis}_{form}".encode(), n, n, 2, 1, ctypes.c_double(0.01), ptr(src), ptr(dst)) == 1
        out.append(dst)
    assert np.any(out[0]) and np.array_equal(*out)


@pytest.mark.parametrize("up", [1, 0])
@pytest.mark.parametrize("warps", [1, 3, 8])
def test_a_cta_publishes_what_its_warps_hold(lanes, warps, up):
    m = np.arange(1, warps + 1, dtype=np.uint64)[::-1].copy()
    v = np.arange(3.0 * warps).reshape(warps, 3) + 0.5
    mo, vo = np.zeros(1, np.uint64), np.zeros(3)
    assert lanes.lanes_publish(warps, up, ptr(m), ptr(v), ptr(mo), ptr(vo)) == 1
    assert mo[0] == warps and np.array_equal(vo, v.sum(0))  # small whole and half numbers: exact


@pytest.mark.parametrize("t64", [0, 1])
@pytest.mark.parametrize("last", [0, 1])
def test_short_control_path_decides_as_the_machine(lanes, t64, last):
    """ctl_fast: the machine's state after an iteration that goes on, and hands over
    whenever the norm accepts, moves the base, is not finite or the counts run out."""
    f = lanes.lanes_ctl
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.c_double] * 4 + [ctypes.c_int] * 2
    tol, base, best = 1e-10, 1e-2, 1e-5
    assert f(t64, 0, 5, 4, best, base, 0.0, tol, 40, last) == 0           # after CI
    up, down = np.nextafter(tol, 1), np.nextafter(tol, 0)
    goes_on = {1e-6: 1, best: 1, 1e-3: 1, up: t64, np.nextafter(1e-6 * base, 1): 1, 1e300: 1,
               tol: 0, down: 0, 0.0: 0, 1e-6 * base: t64, 1.1e300: 0, np.inf: 0, np.nan: 0}
    for nrm, on in goes_on.items():
        assert f(t64, 1, 5, 4, best, base, nrm, tol, 40, last) == (0 if on else 1), nrm
    assert f(t64, 1, 5, 4, best, base, 0.0, 0.0, 40, last) == 1           # tol = 0
    for ev in range(10, 20):                                              # stagnation: FP32 only
        assert f(t64, 1, ev, 4, best, base, 1e-4, tol, 40, last) == (0 if t64 or ev + 1 - 4 < 12 else 1)
    assert f(t64, 1, 38, 37, best, base, 1e-4, tol, 40, last) == 0        # max_iter
    assert f(t64, 1, 39, 38, best, base, 1e-4, tol, 40, last) == 1
    assert f(t64, 1, 61, 60, best, base, 1e-4, tol, 100, last) == 0       # slots
    assert f(t64, 1, 62, 61, best, base, 1e-4, tol, 100, last) == 1
