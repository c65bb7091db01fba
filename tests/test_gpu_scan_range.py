"""Diffusion and growth beyond the range that the scan of the 2-D implicit solve
resolves: such proposals get the oracle's answer, and so do ordinary ones that
share their launch."""
import numpy as np
import pytest
import torch

import oracle
import paper_1605_04718_gb300 as rd
import rd_synth
from tests import gpu_helpers as H
from tests.test_gpu_growing_domain import MODEL5

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
TRUE4 = [0.1, 0.9, 10.0, 200.0]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1605_04718_gb300 import build
    build.build()
    oracle.build()
    rd.load()


def _check(ds, rows, tol, growth=0, kernel=rd.RD_KERNEL_DEFAULT, fill=True):
    """Solves `rows` repeated until the proposals of a grid of N <= 64 fill every CTA
    (so that they share CTAs) and compares every one with its row's oracle solve."""
    n = ds["n"]
    cta = (128 // n) ** 2 if fill and n <= 64 else 0  # proposals a CTA holds
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count
    reps = max(1, -(-cta * sms // len(rows)))
    B = reps * len(rows)
    p = H.gpu_problem([ds], solver=rd.RD_SOLVER_AUTO, growth=growth,
                      model=MODEL5 if growth else H.LOGN4)
    rd.rd_set_size_kernel(p, 0, kernel)
    th = torch.tensor(np.tile(rows, (reps, 1)), dtype=torch.float64, device=DEV)
    phi = torch.zeros(B, dtype=torch.float64, device=DEV)
    st = torch.zeros(B, dtype=torch.int32, device=DEV)
    fl = torch.zeros((B, 2, n, n), dtype=torch.float32, device=DEV)
    rd.rd_evaluate_batch(p, th, phi, st, fields=fl)
    rd.rd_sync(p)
    rd.rd_problem_destroy(p)
    st = st.reshape(reps, len(rows)).cpu().numpy()
    fl = fl.reshape(reps, len(rows), -1)
    P = H.oracle_problem(ds)
    for i, row in enumerate(rows):
        po, so, uo, vo = P.forward(list(row) + [0.0] * (5 - len(row)))
        assert np.all(st[:, i] == so), (i, np.unique(st[:, i]), so)
        if not so:
            want = torch.tensor(np.stack([uo, vo]).ravel(), device=DEV)
            err = float(((fl[:, i].double() - want).norm(dim=1) / want.norm()).max())
            assert err < tol, (i, err)


def _draws(n):
    return rd_synth.lognormal_draws(TRUE4, [0.1] * 4, 9, seed=n)


# 7 steps of rows solved to at most 2^-24 (4 N + 16) of deviations from the mean that
# are below a tenth of the fields: 2.2e-5 at N = 128, 2.2e-6 of the fields
@pytest.mark.parametrize("n", [16, 32, 48, 64, 80, 128])
def test_fast_diffusion_and_its_neighbours(n):
    ds = H.small_dataset(n, 7, seed=n)
    theta = _draws(n)
    theta[1, 2], theta[4, 2], theta[6, 2], theta[7, 2] = 1e16, 1e12, 1e7, 1e30
    _check(ds, theta, 1e-5)


@pytest.mark.parametrize("n", [16, 32, 64])
def test_a_collapsing_domain_leaves_its_neighbours_alone(n):
    """alpha = 1 + 2 tau r = 0.02 without a reaction: the fields grow fiftyfold each step,
    and the scanned values of the second step leave the FP16 range although the
    reaction's (49) do not."""
    ds = H.small_dataset(n, 7, seed=n)
    theta = np.column_stack([_draws(n), np.full(9, 0.01)])
    theta[2, 3:] = 0.0, -1960.0
    _check(ds, theta, 1e-5, growth=1)


# rounding of a step acts on a uniform state that contracts by 1 % or more per step:
# a hundred times 2^-24 (4 N + 16) of the deviation
def test_long_shrinking_and_growing_runs():
    """|2 r T| of 30 to 200: the domain's factors pass the scan's limit on the way, or
    leave no diffusion at all."""
    ds = H.small_dataset(32, 2000, seed=32)
    theta = np.column_stack([np.tile(TRUE4, (27, 1)), np.full(27, 0.01)])
    theta[1, 4], theta[7, 4], theta[13, 4], theta[19, 4], theta[24, 4] = -30.0, -45.0, -50.0, 60.0, 200.0
    _check(ds, theta, 1e-3, growth=1)


# as the first test; four FP32 transforms instead of the elimination
@pytest.mark.parametrize("n", [16, 32, 64, 96, 128])
def test_fast_diffusion_on_the_cuda_cores(n):
    ds = H.small_dataset(n, 7, seed=n)
    theta = _draws(n)
    theta[1, 2], theta[4, 2], theta[6, 2], theta[7, 2] = 1e16, 1e12, 1e7, 1e30
    _check(ds, theta, 1e-5, kernel=rd.RD_KERNEL_SIMT, fill=False)
