"""The FP64 line transforms in 64-bit fixed point (csrc/fx.cuh), through the CPU
emulation of the kernels: their error against an extended-precision DFT is no
larger than that of a plain radix-2 FFT in FP64, over the line lengths and the
kinds of data the passes meet; lines of zeros, of very small and very large
numbers; a NaN or an infinity makes the line NaN."""
import numpy as np
import pytest

from paper_2204_07247_gb300 import pagd


@pytest.fixture(scope="module")
def emu():
    return pagd.load_emulation()


def fft_fp64(x):
    """Radix-2 Stockham FFT in FP64 along the last axis (twiddles rounded once)."""
    n = x.shape[-1]
    a, ns = x.astype(np.complex128), 1
    while ns < n:
        nb = n // 2
        j = np.arange(nb)
        jm = j % ns
        ang = -np.pi * jm.astype(np.longdouble) / ns
        w = (np.cos(ang) + 1j * np.sin(ang)).astype(np.complex128)
        u, v = a[..., :nb], a[..., nb:] * w
        out = np.empty_like(a)
        d = (j - jm) * 2 + jm
        out[..., d], out[..., d + ns] = u + v, u - v
        a, ns = out, 2 * ns
    return a


def dft_long(x):
    """DFT along the last axis in extended precision."""
    n = x.shape[-1]
    k = np.arange(n)
    pi = np.longdouble(np.pi) + np.longdouble(1.2246467991473532e-16)
    ang = -2 * pi * ((np.outer(k, k) % n).astype(np.longdouble)) / n
    return x.astype(np.clongdouble) @ (np.cos(ang) + 1j * np.sin(ang))


def data(kind, n, rng):
    if kind == "field":
        return 0.1 + 0.05 * rng.uniform(-1, 1, n)
    if kind == "noise":
        return rng.standard_normal(n)
    if kind == "smooth":
        x = np.arange(n[1]) / n[1]
        return np.stack([np.sin(2 * np.pi * (i + 1) * x) + 0.1 * np.cos(2 * np.pi * 3 * x + i) for i in range(n[0])])
    if kind == "spike":
        u = 1e-13 * rng.standard_normal(n)
        u[:, 3] = 1.7
        return u
    return rng.standard_normal(n) * np.exp(-0.3 * np.arange(n[1]))  # steep


@pytest.mark.parametrize("kind", ["field", "noise", "smooth", "spike", "steep"])
@pytest.mark.parametrize("m", [8, 16, 32, 64, 128, 256, 512])
def test_error_no_larger_than_an_fp64_fft(emu, kind, m):
    """Rows of length m, columns of length 8: the 2D transform against the
    extended-precision one.  The FP64 side is transformed the same way; its rms
    error estimates the rounding level, and a sample of 8 rows estimates it to
    about 1 / sqrt(8 m) (at most 13%), so the bound is 1.2 times it."""
    n = (8, m)
    S = pagd.Solver("pfc", n, (3.0, 5.0), 0.1, lib=emu)
    e = f = 0.0
    for seed in range(8):
        u = data(kind, n, np.random.default_rng(seed))
        sp = S.fft_r2c(u)
        got = sp[..., 0] + 1j * sp[..., 1]
        ref = dft_long(dft_long(u).T).T
        h = m // 2 + 1
        fp = fft_fp64(fft_fp64(u)[:, :h].T).T
        nrm = np.linalg.norm(ref[:, :h].astype(np.complex128))
        e += float(np.linalg.norm((got - ref[:, :h]).astype(np.complex128)) / nrm) ** 2
        f += float(np.linalg.norm((fp - ref[:, :h]).astype(np.complex128)) / nrm) ** 2
    # one rounding of the result to double is the least either can have
    floor = 8 * (2.0 ** -53 / np.sqrt(3)) ** 2
    assert e <= 1.2 ** 2 * max(f, floor), (np.sqrt(e / 8), np.sqrt(f / 8))


@pytest.mark.parametrize("n", [(16, 64), (128, 128), (32, 512)])
def test_ranges_and_non_finite_lines(emu, n):
    S = pagd.Solver("pfc", n, (3.0, 5.0), 0.1, lib=emu)
    assert not np.any(S.fft_r2c(np.zeros(n)))
    base = S.fft_r2c(0.1 + 0.05 * np.random.default_rng(1).uniform(-1, 1, n))
    for p in (-900, 900):  # scaling by a power of two is exact
        u = (0.1 + 0.05 * np.random.default_rng(1).uniform(-1, 1, n)) * 2.0 ** p
        assert np.array_equal(S.fft_r2c(u) * 2.0 ** -p, base)
        assert np.array_equal(S.fft_c2r(S.fft_r2c(u)) * 2.0 ** -p, S.fft_c2r(base.copy()))
    for bad in (np.nan, np.inf, -np.inf):
        u = np.zeros(n)
        u[3, 2] = bad
        assert np.all(np.isnan(S.fft_r2c(u)))


@pytest.mark.parametrize("n", [(64, 64), (128, 64), (64, 128)])
def test_pair_passes_match_the_warp_passes(emu, monkeypatch, n):
    """The FCH staged passes of two warps per unit and the lines shared by a CTA
    (PAGD_COOP=1) against one warp per unit: two solves accepted at
    ||d|| <= tol differ by at most about 2 tol / (1 - q), q <= 0.9: 20 tol."""
    tol, out = 1e-8, []
    rng = np.random.default_rng(3)
    u0 = -0.3 + 0.05 * rng.uniform(-1, 1, n)
    for coop in ("0", "1"):
        monkeypatch.setenv("PAGD_COOP", coop)
        S = pagd.Solver("fch", n, tuple(v * 4 * np.pi / 256 for v in n), 0.1, 0.1, 0.1, scheme="bdf2",
                        precision="fp32_mixed", lib=emu)
        assert S.launch_info()["coop"] == int(coop) and S.launch_info()["staged"]
        S.set_state(u0)
        o = S.empty_field()
        S.run(1e-3, 2, tol, o)
        out.append(o.copy())
    assert np.abs(out[0] - out[1]).max() <= 20 * tol


@pytest.mark.parametrize("n", [(64, 64), (128, 64)])
def test_pair_passes_take_as_many_evaluations(emu, monkeypatch, n):
    """An exact base evaluation accepts every step, so that a wrong iteration pass
    costs evaluations rather than accuracy: the forms differ by rounding, one
    evaluation a step at most."""
    u0, its = -0.3 + 0.05 * np.random.default_rng(3).uniform(-1, 1, n), []
    for coop in ("0", "1"):
        monkeypatch.setenv("PAGD_COOP", coop)
        S = pagd.Solver("fch", n, tuple(v * 4 * np.pi / 256 for v in n), 0.1, 0.1, 0.1, scheme="bdf2",
                        precision="fp32_mixed", lib=emu)
        S.set_state(u0)
        its.append(np.array(S.run(1e-3, 3, 1e-8, S.empty_field())[0]))
    assert np.abs(its[0] - its[1]).max() <= 1, its
