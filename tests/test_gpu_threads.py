"""Two host threads with problems of different sizes: their calls launch the same
kernels with different amounts of shared memory, and none may change what the
other's launch may take."""
import threading

import numpy as np
import pytest
import torch

from paper_2204_07247_gb300 import inputs as I
from paper_2204_07247_gb300 import pagd
from paper_2204_07247_gb300 import sno as SB

pytestmark = pytest.mark.gpu


def both(jobs, times):
    errors, gate = [], threading.Barrier(len(jobs))

    def loop(job):
        gate.wait()
        try:
            for _ in range(times):
                job()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
    ts = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors


def test_networks_of_different_sizes():
    jobs, want = [], []
    for n, C in (((16, 512), 17), ((64, 512), 32)):
        net = SB.SNO(n, channels=C, layers=2, modes=(8, 32), batch=1, seed=3)
        un = torch.from_numpy(I.noisy_field(n, -0.3, 0.3, 1)[None]).cuda()
        um, out = un + 0.01, torch.empty_like(un)
        ref = net.predict(un, um, 1.0, 20.0, 0.02).clone()
        jobs.append(lambda net=net, un=un, um=um, out=out: net.predict(un, um, 1.0, 20.0, 0.02, out))
        want.append((out, ref))
    both(jobs, 300)
    for out, ref in want:
        assert torch.equal(out, ref)


def test_solvers_of_different_models():
    jobs = []
    for model, eta in (("pfc", 0.0), ("fch", 0.1)):
        S = pagd.Solver(model, (64, 64), (20.0, 20.0), 0.1, eta, eta, scheme="bdf2", precision="fp32_mixed")
        u = torch.from_numpy(I.noisy_field((64, 64), 0.1, 0.05, 1)).cuda()
        o = S.empty_field()

        def job(S=S, u=u, o=o):
            S.set_state(u)
            _, res = S.run(1e-3, 1, 1e-8, o)
            assert np.all(res <= 1e-8)
        jobs.append(job)
    both(jobs, 100)
