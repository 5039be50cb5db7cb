"""The number helpers of csrc/fx.cuh and solver.cuh against IEEE arithmetic: on
the CPU through the host build of the same source, and on the GPU (marked gpu).

Conversions are exact or rounded to nearest even, so they have to agree bit for
bit, except for subnormal FP32 results, which are rounded twice.  The reciprocal is one rounding of x0 (1 + e + e^2) with |e| <= 2^-21, the
inner sum's rounding being 2^-53 of e: at most 0.5 + 2^-10 ulp, and 0.501 with the
rounding of the check itself; the quotient's correction leaves as much."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2204_07247_gb300", "csrc")


class Host:
    def __init__(self, d):
        so = os.path.join(d, "libarith.so")
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-DPAGD_EMU", "-ffp-contract=off", "-w", "-x", "c++", "-I", CSRC,
                               "-fPIC", "-shared", "-o", so, os.path.join(HERE, "lanes", "arith.cu")])
        self.lib = ctypes.CDLL(so)

    warp = 1

    def __call__(self, fn, out_type, *arrays, n=None, extra=()):
        out = np.zeros(n or len(arrays[0]), out_type)
        keep = [np.ascontiguousarray(a) for a in arrays]
        args = [ctypes.c_void_p(a.ctypes.data) for a in keep]
        assert getattr(self.lib, fn)(*args, ctypes.c_void_p(out.ctypes.data), ctypes.c_longlong(len(out)), *extra) == 0
        return out


class Device:
    def __init__(self, d):
        from paper_2204_07247_gb300 import build as B
        so = os.path.join(d, "libarith_gpu.so")
        subprocess.check_call([B.nvcc(), "-gencode", B.GENCODE, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", CSRC,
                               "-shared", "-o", so, os.path.join(HERE, "lanes", "arith.cu")])
        self.lib = ctypes.CDLL(so)

    warp = 32

    def __call__(self, fn, out_type, *arrays, n=None, extra=()):
        import torch
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]
        out = torch.from_numpy(np.zeros(n or len(arrays[0]), out_type)).cuda()
        torch.cuda.synchronize()
        args = [ctypes.c_void_p(t.data_ptr()) for t in dev]
        assert getattr(self.lib, fn)(*args, ctypes.c_void_p(out.data_ptr()), ctypes.c_longlong(len(out)), *extra) == 0
        return out.cpu().numpy()


@pytest.fixture(scope="module", params=["host", pytest.param("device", marks=pytest.mark.gpu)])
def run(request, tmp_path_factory):
    return (Host if request.param == "host" else Device)(str(tmp_path_factory.mktemp("arith")))


def doubles(seed=0):
    """every exponent with random significands, values half way between two FP32
    numbers and next to them, the limits of both formats, zeros, infinities, NaN"""
    r = np.random.default_rng(seed)
    e = np.repeat(np.arange(2047, dtype=np.uint64), 24)
    any_e = (e << np.uint64(52)) | r.integers(0, 2 ** 52, e.size, dtype=np.uint64)
    f = np.concatenate([(e & np.uint64(255)) << np.uint64(23) | r.integers(0, 2 ** 23, e.size, dtype=np.uint64),
                        np.arange(0, 40, dtype=np.uint64), 0x7fffff + np.arange(-20, 20).astype(np.uint64)])
    f = f.astype(np.uint32).view(np.float32)
    f = f[np.isfinite(f)].astype(np.float64)
    up = np.nextafter(f.astype(np.float32), np.float32(np.inf)).astype(np.float64)
    tie = np.where(np.isfinite(up), (f + up) / 2, f)
    edge = np.array([0.0, np.inf, np.nan, 2.0 ** -1074, 2.0 ** -1022, 2.0 ** -149, 2.0 ** -150, 2.0 ** -126, 2.0 ** 127,
                     2.0 ** 128, np.finfo(np.float32).max, 1.0, 1 / 3])
    x = np.concatenate([any_e.view(np.float64), f, tie, np.nextafter(tie, np.inf), np.nextafter(tie, -np.inf), edge,
                        np.nextafter(edge, 0), np.nextafter(edge, np.inf)])
    return np.concatenate([x, -x])


def same(a, b):
    """bit for bit, any NaN for a NaN"""
    n = np.isnan(b)
    assert np.array_equal(np.isnan(a), n)
    u = np.uint32 if a.dtype == np.float32 else np.uint64
    bad = np.flatnonzero(a.view(u)[~n] != b.view(u)[~n])
    assert bad.size == 0, (a[~n][bad[:4]], b[~n][bad[:4]])


def ulps(got, ref):
    """|got - ref| in units of the last place of ref (extended precision)"""
    u = np.spacing(np.abs(ref.astype(np.float64)))
    return np.abs((got.astype(np.longdouble) - ref) / u)


def normals(seed=1):
    """positive normal numbers whose reciprocals are normal, and significands next to 1 and 2"""
    r = np.random.default_rng(seed)
    e = np.repeat(np.arange(1, 2042, dtype=np.uint64), 64)
    m = r.integers(0, 2 ** 52, e.size, dtype=np.uint64)
    m[::8] >>= np.uint64(40)
    m[1::8] |= np.uint64(0xffffff0000000)
    return ((e << np.uint64(52)) | m).view(np.float64)


def test_reciprocal(run):
    x = normals()
    assert ulps(run("arith_rcp", np.float64, x), 1 / x.astype(np.longdouble)).max() <= 0.501
    rest = doubles()
    rest = rest[(rest <= 0) | (rest >= 2.0 ** 1020) | (np.abs(rest) < 2.0 ** -1022) | np.isnan(rest)]
    with np.errstate(all="ignore"):  # every other number: the division
        same(run("arith_rcp", np.float64, rest), 1 / rest)


def test_quotient(run):
    x = normals()
    x = x[(x > 2.0 ** -900) & (x < 2.0 ** 900)]
    n = np.random.default_rng(2).uniform(-3, 3, x.size) * 2.0 ** np.random.default_rng(3).integers(-60, 60, x.size)
    got = run("arith_div", np.float64, np.stack([n, x], 1).ravel()).reshape(-1, 2)
    lx = x.astype(np.longdouble)
    assert ulps(got[:, 0], n / lx).max() <= 0.501 and ulps(got[:, 1], 1 / lx).max() <= 0.501
    pairs = np.array([[1.0, np.inf], [0.0, 3.0], [2.0, 0.0], [3.0, -7.0], [1.0, 5e-324], [np.nan, 1.0], [1.0, np.nan]])
    with np.errstate(all="ignore"):
        same(run("arith_div", np.float64, pairs.ravel()).reshape(-1, 2)[:, 0].copy(), pairs[:, 0] / pairs[:, 1])


def test_preconditioner_factors(run):
    """1 / (M kappa): two roundings; L: its sum, positive terms but one, against the
    sum of their magnitudes: six roundings of half an ulp."""
    kap = np.concatenate([10.0 ** np.random.default_rng(4).uniform(-12, 16, 4000), 10.0 ** np.arange(17, 120, 7.0)])
    got = run("arith_pre", np.float64, np.concatenate([kap, np.zeros(kap.size)])).reshape(-1, 2)
    k, M = kap.astype(np.longdouble), np.longdouble(1.3)
    assert ulps(got[:, 0], 1 / (M * k)).max() <= 1.01 * 2  # relative 2 x 2^-53, up to 2 ulp of a smaller significand
    terms = np.stack([4 / (M * k), np.full(kap.size, np.longdouble(0.7)), -2 * k, k * k])
    assert (np.abs(got[:, 1] - terms.sum(0)) / np.abs(terms).sum(0)).max() <= 6 * 2.0 ** -53


@pytest.mark.parametrize("kind", ["same sign", "mixed", "cancelling", "wide"])
def test_sum_no_less_exact_than_fp64(run, kind):
    """64 sums of 32 x 400 (host: 400) values: within a last place of the
    exact sum plus 2^-70 of the magnitudes, which is less than FP64 leaves"""
    m, n = 400, 64 * run.warp
    r = np.random.default_rng(5)
    a = r.uniform(0.5, 1, (64, run.warp * m))
    if kind != "same sign":
        a *= r.choice([-1, 1], a.shape)
    if kind == "cancelling":  # pairs of opposite values and a small rest
        h = a.shape[1] // 2
        a[:, h:] = -a[:, :h][:, ::-1]
        a[:, ::7] += 1e-4 * r.uniform(-1, 1, a[:, ::7].shape)
    if kind == "wide":
        a *= 2.0 ** r.integers(-60, 60, a.shape)
    a = a.astype(np.float32)
    got = run("arith_sum", np.float64, a.ravel(), np.arange(n, dtype=np.int32), n=n, extra=(ctypes.c_int(m),))
    err = err64 = 0.0
    for i in range(64):
        x = a[i].astype(np.float64)
        ref, mag = math.fsum(x), math.fsum(np.abs(x))
        e = [float(abs(Fraction(float(g)) - Fraction(ref))) for g in got[i * run.warp:(i + 1) * run.warp]]
        assert max(e) <= np.spacing(abs(ref)) + 2.0 ** -70 * mag  # (fsum itself is rounded)
        err = max(err, max(e) / mag)
        err64 = max(err64, abs(float(np.cumsum(x)[-1]) - ref) / mag)
    assert err <= err64


def test_sum_of_infinities(run):
    a = np.ones((run.warp, 4), np.float32)
    for bad, want in ((np.inf, np.inf), (-np.inf, -np.inf), (np.nan, np.nan)):
        a[0, 1] = bad
        got = run("arith_sum", np.float64, a.ravel(), np.arange(run.warp, dtype=np.int32), n=run.warp, extra=(ctypes.c_int(4),))
        same(got, np.full(run.warp, want))


def test_fp64_to_fp32(run):
    x = doubles()
    with np.errstate(over="ignore"):
        want = x.astype(np.float32)
    got = run("arith_f32", np.float32, x)
    sub = np.abs(x) < 2.0 ** -126
    same(got[~sub], want[~sub])
    # subnormal results: rounded at 24 bits, then to the last place 2^-149
    exact = x[sub].astype(np.longdouble)
    assert np.array_equal(np.signbit(got[sub]), np.signbit(x[sub]))
    assert (np.abs(got[sub] - exact) <= 2.0 ** -150 + np.abs(exact) * 2.0 ** -24).all()


def test_fp32_to_fp64(run):
    with np.errstate(over="ignore"):
        x = np.unique(doubles().astype(np.float32).view(np.uint32)).view(np.float32)
    same(run("arith_f64", np.float64, x), x.astype(np.float64))
