"""The number helpers of csrc/fx.cuh against IEEE arithmetic: on the CPU through
the host build of the same source, and on the GPU (marked gpu).  Conversions are
exact or rounded to nearest even, so they have to agree bit for bit."""
import ctypes
import os
import subprocess

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

    def __call__(self, fn, out_type, *arrays):
        out = np.zeros(len(arrays[0]), out_type)
        keep = [np.ascontiguousarray(a) for a in arrays]
        args = [ctypes.c_void_p(a.ctypes.data) for a in keep]
        assert getattr(self.lib, fn)(*args, ctypes.c_void_p(out.ctypes.data), ctypes.c_longlong(len(out))) == 0
        return out


class Device:
    def __init__(self, d):
        from paper_2204_07247_gb300 import build as B
        so = os.path.join(d, "libarith_gpu.so")
        subprocess.check_call([B.nvcc(), "-gencode", B.GENCODE, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", CSRC,
                               "-shared", "-o", so, os.path.join(HERE, "lanes", "arith.cu")])
        self.lib = ctypes.CDLL(so)

    def __call__(self, fn, out_type, *arrays):
        import torch
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]
        out = torch.from_numpy(np.zeros(len(arrays[0]), out_type)).cuda()
        torch.cuda.synchronize()
        args = [ctypes.c_void_p(t.data_ptr()) for t in dev]
        assert getattr(self.lib, fn)(*args, ctypes.c_void_p(out.data_ptr()), ctypes.c_longlong(len(out))) == 0
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


def test_fp64_to_fp32(run):
    x = doubles()
    with np.errstate(over="ignore"):
        same(run("arith_f32", np.float32, x), x.astype(np.float32))


def test_fp32_to_fp64(run):
    with np.errstate(over="ignore"):
        x = np.unique(doubles().astype(np.float32).view(np.uint32)).view(np.float32)
    same(run("arith_f64", np.float64, x), x.astype(np.float64))
