"""The tensor-core solve at every grid size and at batch sizes around the number
of proposals a CTA holds, against the FP64 oracle; proposals whose solve
diverges beside ones that do not; parameters outside the scan's range."""
import numpy as np
import pytest
import torch

import oracle
import paper_1605_04718_gb300 as rd
import rd_synth
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
TRUE4 = [0.1, 0.9, 10.0, 200.0]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1605_04718_gb300 import build
    build.build()
    oracle.build()
    rd.load()


def _eval(p, theta, n):
    B = len(theta)
    th = torch.tensor(theta, dtype=torch.float64, device=DEV)
    phi = torch.zeros(B, dtype=torch.float64, device=DEV)
    st = torch.zeros(B, dtype=torch.int32, device=DEV)
    fl = torch.zeros((B, 2, n, n), dtype=torch.float32, device=DEV)
    rd.rd_evaluate_batch(p, th, phi, st, fields=fl)
    rd.rd_sync(p)
    return phi.cpu().numpy(), st.cpu().numpy(), fl.double().cpu().numpy()


# batches: one proposal; one CTA's worth per SM and one more; a partly filled CTA
@pytest.mark.parametrize("n,batch", [(16, 1), (16, 37), (16, 152 * 64 + 1), (32, 3), (32, 152 * 16 + 5),
                                     (48, 2), (48, 609), (64, 1), (64, 305), (64, 611), (80, 3),
                                     (96, 153), (112, 2), (128, 153)])
@pytest.mark.parametrize("steps", [7])
def test_every_size_matches_the_oracle(n, batch, steps):
    """Fields within 7 steps of two split-FP16 stages (operands to 2^-22, sums
    rounded toward zero to 2^-23 of the largest partial sum) and one scan: below
    40 x 2^-22 = 1e-5 relative."""
    ds = H.small_dataset(n, steps, seed=n + batch, obs_frac=(3 / 7, 1.0))
    p = H.gpu_problem([ds], solver=rd.RD_SOLVER_AUTO)
    theta = rd_synth.lognormal_draws(TRUE4, [0.15] * 4, batch, seed=batch)
    phi, st, fl = _eval(p, theta, n)
    rd.rd_problem_destroy(p)
    assert np.all(st == 0) and np.all(np.isfinite(phi))
    P = H.oracle_problem(ds)
    for i in sorted({0, batch // 2, batch - 1, min(batch - 1, 33)}):
        po, so, uo, vo = P.forward(list(theta[i]) + [0.0])
        assert so == 0
        assert H.rel_l2(fl[i], np.stack([uo, vo])) < 1e-5, i
        assert abs(phi[i] - po) <= 1e-4 * po, i


@pytest.mark.parametrize("n", [16, 32, 48, 64, 96])
def test_a_diverging_solve_leaves_its_neighbours_alone(n):
    """Every third proposal blows up (gamma 2000 times too large): status
    RD_P_NONFINITE and Phi = inf there, the oracle's fields everywhere else."""
    ds = H.small_dataset(n, 40, seed=3 * n)
    p = H.gpu_problem([ds], solver=rd.RD_SOLVER_AUTO)
    theta = rd_synth.lognormal_draws(TRUE4, [0.1] * 4, 25, seed=n)
    theta[::3, 3] = 4e5
    phi, st, fl = _eval(p, theta, n)
    rd.rd_problem_destroy(p)
    P = H.oracle_problem(ds)
    for i in range(25):
        po, so, uo, vo = P.forward(list(theta[i]) + [0.0])
        assert st[i] == so == (rd.RD_P_NONFINITE if i % 3 == 0 else 0)
        if so:
            assert np.isinf(phi[i])
        else:
            assert H.rel_l2(fl[i], np.stack([uo, vo])) < 1e-5


@pytest.mark.parametrize("n", [16, 32, 64, 80, 128])
def test_parameters_outside_the_scan_match_the_cuda_core_kernel(n):
    """d <= 0 (the tridiagonal factors are not positive): solved by elimination;
    the transforms of the CUDA-core kernel take any d."""
    ds = H.small_dataset(n, 4, seed=n)
    theta = rd_synth.lognormal_draws(TRUE4, [0.1] * 4, 9, seed=n)
    theta[1, 2], theta[4, 2], theta[5, 2], theta[8, 2] = -0.02, 0.0, -0.01, float("nan")
    out = {}
    p = H.gpu_problem([ds], solver=rd.RD_SOLVER_AUTO)
    for k in (rd.RD_KERNEL_DEFAULT, rd.RD_KERNEL_SIMT):
        rd.rd_set_size_kernel(p, 0, k)
        out[k] = _eval(p, theta, n)
    rd.rd_problem_destroy(p)
    (pa, sa, fa), (pb, sb, fb) = out.values()
    assert np.array_equal(sa, sb) and sa[8] == rd.RD_P_NONFINITE
    for i in range(8):
        assert sa[i] == 0
        assert H.rel_l2(fa[i], fb[i]) < 2e-5, i


def test_chains_over_several_sizes_hold_the_phi_of_their_state():
    """One launch per size, started before the previous one ends, inside the
    captured step: every chain's stored Phi is that of its own state and size."""
    dss = [H.small_dataset(n, 30, seed=n, sigma=0.3) for n in (128, 32, 80)]
    p = H.gpu_problem(dss, solver=rd.RD_SOLVER_AUTO)
    C = 23
    size_idx = np.arange(C) % 3
    theta0 = rd_synth.lognormal_draws(TRUE4, [0.05] * 4, C, seed=5)
    c = rd.rd_chains_create(p, theta0, 7, [0.02] * 4, size_idx=size_idx, capacity=8)
    for _ in range(3):
        rd.rd_chains_run(c, 2)
    samples, counters = rd.rd_chains_read_samples(c, 6, 4, C)
    th, phi = rd.rd_chains_get_state(c, 4, C)
    assert counters[2] > 0 and np.array_equal(samples[-1].T, th)
    got, st = rd.rd_evaluate_batch_host(p, th, size_idx=size_idx)
    rd.rd_chains_destroy(c)
    rd.rd_problem_destroy(p)
    assert np.all(st == 0) and np.all(np.abs(got - phi) <= 1e-12 * phi)
