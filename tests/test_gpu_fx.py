"""GPU: the fixed-point FP64 lines in every form a launch picks (a warp per
line, lines shared by a CTA, one unit per CTA with two CTAs on an SM), the
passes of two warps per unit, and the network's tiles over their line lengths.

Tolerances.  A transform is two or three passes, each with at most the rounding
of an FP64 FFT (2^-53 sqrt(log2 n) relative, 3.4e-16 for 512 points), against
numpy's FFT with as much: 1e-15 covers sqrt(6) of them.  Two solves accepted at
||d|| <= tol differ by at most about 2 tol / (1 - q) with a contraction q <= 0.9
per evaluation: 20 tol.  The network: 1e-5 relative on the guess and 1e-4 on the
gradient, as in test_gpu_sno.py."""
import math

import numpy as np
import pytest
import torch

from oracle import sno_oracle as SO
from paper_2204_07247_gb300 import inputs as I
from paper_2204_07247_gb300 import pagd
from paper_2204_07247_gb300 import sno as SB

pytestmark = pytest.mark.gpu

GRIDS = [(8, 8), (16, 512), (512, 8), (32, 32), (64, 64), (64, 256), (128, 128), (256, 512), (512, 512), (8, 16, 32),
         (64, 128, 64), (128, 128, 128), (256, 64, 256)]


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("coop", ["0", "1", None])
@pytest.mark.parametrize("n", GRIDS)
def test_transforms_in_every_form(monkeypatch, n, coop):
    if coop is not None:
        monkeypatch.setenv("PAGD_COOP", coop)
    S = pagd.Solver("pfc", n, (3.0,) * len(n), 0.1)
    u = 0.1 + 0.05 * np.random.default_rng(sum(n)).uniform(-1, 1, n)
    sp = S.fft_r2c(dev(u)).cpu().numpy()
    ref = np.fft.rfftn(u)
    assert np.linalg.norm(sp[..., 0] + 1j * sp[..., 1] - ref) <= 1e-15 * np.linalg.norm(ref)
    back = S.fft_c2r(dev(sp)).cpu().numpy()
    assert np.linalg.norm(back - u) <= 1e-15 * np.linalg.norm(u)


@pytest.mark.parametrize("model,n", [("fch", (64, 64)), ("fch", (128, 64)), ("fch", (64, 512)), ("fch", (256, 256)),
                                     ("fch", (512, 512)), ("pfc", (512, 512)), ("pfc", (64, 256)), ("pfc", (512, 128))])
def test_small_grid_forms_agree(monkeypatch, model, n):
    """FP32-mixed steps with and without the shared forms (PAGD_COOP): pairs of
    warps (FCH), shared FP32 lines, one unit per CTA (512^2), staged rectangles."""
    h = math.pi / 4 if model == "pfc" else 4 * math.pi / 256
    tol, out = 1e-10, []
    for coop in ("0", "1"):
        monkeypatch.setenv("PAGD_COOP", coop)
        eta = 0.1 if model == "fch" else 0.0
        S = pagd.Solver(model, n, tuple(h * v for v in n), 0.1, eta, eta, scheme="bdf2", precision="fp32_mixed")
        S.set_state(dev(I.noisy_field(n, -0.3 if model == "fch" else 0.1, 0.05, 5)))
        u = S.empty_field()
        _, res = S.run(1e-3 if model == "fch" else 0.1, 3, tol, u)
        assert np.all(res <= tol)
        out.append(u.cpu().numpy())
    assert np.abs(out[0] - out[1]).max() <= 20 * tol


def test_non_finite_state_is_an_error():
    for bad in (np.nan, np.inf):
        for n in ((64, 64), (512, 512)):
            u = I.noisy_field(n, 0.1, 0.05, 1)
            u[3, 4] = bad
            S = pagd.Solver("pfc", n, (20.0, 20.0), 0.1, scheme="mp")
            S.set_state(dev(u))
            with pytest.raises(pagd.PagdError) as e:
                S.step(S.empty_field(), 0.1, 1e-10)
            assert e.value.status == 6


@pytest.mark.parametrize("n,C,L,modes,B", [((8, 8), 3, 2, (4, 3), 2), ((16, 16), 5, 1, (6, 8), 3), ((8, 32), 32, 2, (4, 16), 2),
                                           ((32, 64), 17, 2, (8, 17), 2), ((16, 128), 16, 3, (16, 16), 2),
                                           ((8, 256), 7, 2, (2, 32), 3), ((32, 512), 16, 2, (16, 16), 2),
                                           ((16, 1024), 20, 2, (8, 5), 2), ((1024, 16), 6, 2, (32, 7), 1)])
def test_network_tiles(n, C, L, modes, B):
    net = SB.SNO(n, channels=C, layers=L, modes=modes, batch=B, seed=3)
    net.params += 0.05 * torch.from_numpy((2 * I.uniform01(7, net.nparams) - 1).astype(np.float32)).cuda()
    un = np.stack([I.noisy_field(n, -0.3, 0.3, b) for b in range(B)])
    um = un + 0.01 * np.stack([I.noisy_field(n, 0.0, 1.0, 50 + b) for b in range(B)])
    tg = un + 0.02 * np.stack([I.noisy_field(n, 0.0, 1.0, 90 + b) for b in range(B)])
    theta = net.params.double().cpu()
    t = torch.from_numpy
    guess = net.predict(dev(un), dev(um), 1.0, 20.0, 0.02).cpu()
    ref, _ = SO.forward(theta, t(un), t(um), 1.0, 20.0, 0.02, C, L, *modes)
    assert torch.linalg.norm(guess - ref) <= 1e-5 * torch.linalg.norm(ref)
    loss, grad = net.loss_grad(dev(un), dev(um), dev(tg), 1.0, 20.0, 0.02)
    rl, rg = SO.loss_and_grad(theta, t(un), t(um), t(tg), 1.0, 20.0, 0.02, C, L, *modes)
    assert abs(loss - rl) <= 1e-5 * abs(rl)
    assert torch.linalg.norm(grad.double().cpu() - rg) <= 1e-4 * torch.linalg.norm(rg)


@pytest.mark.parametrize("model,n", [("fch", (64, 64)), ("fch", (64, 512)), ("fch", (256, 256)), ("fch", (512, 512)),
                                     ("pfc", (512, 512)), ("pfc", (64, 256))])
def test_small_grid_forms_take_as_many_evaluations(monkeypatch, model, n):
    """The states agree as long as the iterations converge at all (an exact base
    evaluation accepts); a wrong iteration pass shows in their number.  The forms
    differ by rounding: one evaluation a step at most, two for a rebase it moves."""
    h, its = math.pi / 4 if model == "pfc" else 4 * math.pi / 256, []
    eta = 0.1 if model == "fch" else 0.0
    for coop in ("0", "1"):
        monkeypatch.setenv("PAGD_COOP", coop)
        S = pagd.Solver(model, n, tuple(h * v for v in n), 0.1, eta, eta, scheme="bdf2", precision="fp32_mixed")
        S.set_state(dev(I.noisy_field(n, -0.3 if model == "fch" else 0.1, 0.05, 5)))
        its.append(np.array(S.run(1e-3 if model == "fch" else 0.1, 3, 1e-10, S.empty_field())[0]))
    assert np.abs(its[0] - its[1]).max() <= 3, its


@pytest.mark.parametrize("n,shared", [((64, 8, 64), 1), ((64, 16, 64), 0), ((128, 8, 128), 0), ((32, 16, 32), 0), ((32, 32, 32), 0),
                                      ((16, 16, 16), 1), ((8, 8, 8), 1)])
def test_3d_grids_share_units_only_in_few_rounds(n, shared):
    """Which of the two forms a 3D grid takes on 152 SMs, and that they agree: the
    tolerance of the transforms above."""
    S = pagd.Solver("pfc", n, (3.0,) * 3, 0.1)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert S.launch_info()["coop"] == shared
    u = 0.1 + 0.05 * np.random.default_rng(sum(n)).uniform(-1, 1, n)
    sp = S.fft_r2c(dev(u)).cpu().numpy()
    ref = np.fft.rfftn(u)
    assert np.linalg.norm(sp[..., 0] + 1j * sp[..., 1] - ref) <= 1e-15 * np.linalg.norm(ref)
