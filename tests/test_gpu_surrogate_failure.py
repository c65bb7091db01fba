"""Failure detection of the surrogate's kernels, tested without a GPU fault: a test aid
leaves the completion of their products unsignalled, the wait limit is set short, and
the launch must end in bounded time with RD_ETIMEOUT and its tensor memory free: the
next call gives the results of a call before the failure."""
import time

import numpy as np
import pytest
import torch

import paper_1605_04718_gb300 as rd
import rd_synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
TRUE4 = [0.1, 0.9, 10.0, 200.0]


@pytest.mark.parametrize("rows", [256, 20096])  # tiles of 32 and of 128 rows
def test_bounded_wait_gives_up_and_the_surrogate_recovers(rows):
    from paper_1605_04718_gb300 import build
    build.build()
    rd.load()
    desc = rd.make_desc(2, [32], 2.5e-4, 10, [0, 1, 2, 3], TRUE4 + [0.0],
                        [rd.RD_PRIOR_LOGNORMAL] * 4, TRUE4, [0.5] * 4, [rd.RD_STEP_LOG] * 4)
    p = rd.rd_problem_create(desc)
    s = rd.rd_surrogate_create(p, 3)
    th = torch.tensor(rd_synth.lognormal_draws(TRUE4, [0.5] * 4, rows, seed=1),
                      dtype=torch.float64, device=DEV)
    target = torch.linspace(-1, 1, rows, device=DEV)
    n = rd.rd_surrogate_get_params(s)[0].size

    def predict():
        phi = torch.zeros(rows, dtype=torch.float64, device=DEV)
        rd.rd_surrogate_predict(s, th, phi)
        return phi

    def grads():
        g = torch.zeros(n, dtype=torch.float32, device=DEV)
        rd.rd_surrogate_loss_grad(s, th, target, g)
        return g

    before = predict(), grads()
    rd.rd_sync(p)
    rd.rd_set_wait_limit(p, 0.05)
    rd.rd_debug_stall_at_step(p, rd.RD_STALL_SURROGATE)
    for call in (predict, grads):
        t0 = time.perf_counter()
        call()
        with pytest.raises(rd.RdError) as ei:
            rd.rd_sync(p)
        assert ei.value.code == rd.RD_ETIMEOUT
        assert time.perf_counter() - t0 < 30.0
    rd.rd_debug_stall_at_step(p, -1)
    rd.rd_set_wait_limit(p, 4.0)
    after = predict(), grads()
    rd.rd_sync(p)
    assert torch.equal(after[0], before[0])
    assert np.array_equal(after[1].cpu().numpy(), before[1].cpu().numpy())
    rd.rd_surrogate_destroy(s)
    rd.rd_problem_destroy(p)
