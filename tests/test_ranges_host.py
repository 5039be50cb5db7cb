"""Grids far from the usual spacing, through the CPU emulation: the FP32 iteration
passes carry wavenumbers up to kappa = 1e13 (their squares are FP32 numbers) and
take as many evaluations there as on an ordinary domain."""
import numpy as np
import pytest

from paper_2204_07247_gb300 import pagd


@pytest.mark.parametrize("n", [(16, 16), (64, 64)])
@pytest.mark.parametrize("model,eta", [("pfc", 0.0), ("fch", 0.1)])
def test_small_domains_iterate_like_ordinary_ones(model, eta, n):
    evals = []
    for L in (0.01, 1e-3, 1e-5):
        S = pagd.Solver(model, n, (L, L), 0.1, eta, eta, scheme="bdf2", precision="fp32_mixed",
                        lib=pagd.load_emulation())
        S.set_state(0.1 + 0.05 * np.random.default_rng(0).uniform(-1, 1, n))
        it, res = S.run(0.1, 2, 1e-10, S.empty_field())
        assert np.all(res <= 1e-10)
        evals.append(np.array(it))
    # every mode but the mean decays at once on each of them: the same steps, up
    # to one evaluation of rounding
    assert max(np.abs(e - evals[0]).max() for e in evals) <= 1, evals


@pytest.mark.parametrize("p", [-1000, -1022, -1040, -1060])
@pytest.mark.parametrize("n", [(8, 8), (16, 128), (256, 32), (8, 512)])
def test_subnormal_lines(n, p):
    """Fields around 2^p: the spectrum is the one of the same numbers scaled up, to
    the last place of a subnormal number: one rounding per point after each of the
    two passes, the first ones summed by the second."""
    S = pagd.Solver("pfc", n, (3.0, 5.0), 0.1, lib=pagd.load_emulation())
    u = (0.1 + np.random.default_rng(1).uniform(-1, 1, n)) * 2.0 ** p
    up = u * 2.0 ** 900 * 2.0 ** (-p - 900)  # exact
    want = S.fft_r2c(up) * 2.0 ** p
    assert np.any(want)
    tol = (n[0] + 1) * 2.0 ** -1074 + 1e-15 * np.abs(want).max()
    assert np.abs(S.fft_r2c(u) - want).max() <= tol
    back = S.fft_c2r(S.fft_r2c(u))
    assert np.abs(back - u).max() <= 3 * tol


@pytest.mark.parametrize("model,eta,size,dt", [("pfc", 0.0, 1e18, 1e-50), ("pfc", 0.0, 5e18, 1e-50), ("fch", 0.1, 1e9, 1e-60)])
def test_sums_of_large_values(model, eta, size, dt):
    """Fields whose averaged-Newton values are FP32 numbers, but not their sum
    over the grid (3 u^2 and about 45 u^4 against 3.4e38)."""
    S = pagd.Solver(model, (64, 64), (20.0, 20.0), 0.1, eta, eta, scheme="bdf2", lib=pagd.load_emulation())
    S.set_state(size * (1 + 0.05 * np.random.default_rng(0).uniform(-1, 1, (64, 64))))
    _, res = S.run(dt, 1, 1e-13 * size, S.empty_field())
    assert np.all(res <= 1e-13 * size)
