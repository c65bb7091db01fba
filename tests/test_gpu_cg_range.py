"""The conjugate-gradient solves over the whole exponent range of FP32 fields: with
gamma = 0 the step is linear in each field, so fields scaled by powers of two
(products of their values under- or overflow FP32) give the scaled result."""
import numpy as np
import pytest
import torch

import paper_1605_04718_gb300 as rd
from tests import gpu_helpers as H

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1605_04718_gb300 import build
    build.build()
    rd.load()


def _diffuse(n, steps, scale, picard):
    rng = np.random.default_rng(n)
    w = rng.uniform(0.5, 1.5, (2, n, n)).astype(np.float32).astype(np.float64)
    w *= np.asarray(scale)[:, None, None]
    desc = rd.make_desc(2, [n], 2.5e-4, steps, fixed=[0.1, 0.9, 10.0, 0.0, 0.0],
                        solver=rd.RD_SOLVER_AUTO, w_max=1e30, **H.LOGN4)
    p = rd.rd_problem_create(desc)
    rd.rd_set_initial_state(p, 0, w[0], w[1])
    rd.rd_set_observations(p, 0, [steps], 3, w[None], 1.0)
    if picard:
        rd.rd_set_scheme(p, rd.RD_SCHEME_PICARD)
    else:
        rd.rd_set_size_kernel(p, 0, rd.RD_KERNEL_CG)
    th = torch.tensor([[0.1, 0.9, 10.0, 0.0]] * 2, dtype=torch.float64, device=DEV)
    phi = torch.zeros(2, dtype=torch.float64, device=DEV)
    st = torch.full((2,), -1, dtype=torch.int32, device=DEV)
    fl = torch.zeros((2, 2, n, n), dtype=torch.float32, device=DEV)
    rd.rd_evaluate_batch(p, th, phi, st, fields=fl)
    rd.rd_sync(p)
    rd.rd_problem_destroy(p)
    return st.cpu().numpy(), fl[1].double().cpu().numpy() / np.asarray(scale)[:, None, None]


# each of 4 steps solves both runs to a relative residual of 1e-6, and the operator is
# at least the identity: 4 x 2 x 1e-6 (relative to the fields, which exceed the deviations)
@pytest.mark.parametrize("n,picard", [(16, False), (64, False), (96, False), (32, True), (80, True)])
@pytest.mark.parametrize("scale", [(2.0**-73, 2.0**73), (2.0**-60, 2.0**62), (2.0**-100, 2.0**80)])
def test_scaled_fields_give_the_scaled_result(n, picard, scale):
    st0, ref = _diffuse(n, 4, (1.0, 1.0), picard)
    st1, got = _diffuse(n, 4, scale, picard)
    assert np.all(st0 == 0) and np.all(st1 == 0)
    for f in range(2):
        assert H.rel_l2(got[f], ref[f]) < 8e-6, f


def test_a_diverging_proposal_is_not_taken_for_an_unconverged_solve():
    """gamma 200 times too large: the fields pass 1e19 on their way out, where products of
    their values overflow FP32 although every system is still solved; the status is
    RD_P_NONFINITE alone, as the oracle's."""
    ds = H.small_dataset(64, 100, seed=64)
    p = H.gpu_problem([ds], solver=rd.RD_SOLVER_AUTO)
    rd.rd_set_size_kernel(p, 0, rd.RD_KERNEL_CG)
    theta = np.tile([0.1, 0.9, 10.0, 200.0], (9, 1))
    theta[::3, 3] = 4e4
    phi, st = rd.rd_evaluate_batch_host(p, theta)
    rd.rd_problem_destroy(p)
    P = H.oracle_problem(ds)
    for i in range(9):
        assert st[i] == P.forward(list(theta[i]) + [0.0])[1]
    assert np.array_equal(np.isinf(phi), theta[:, 3] > 1e3)
