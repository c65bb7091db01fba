"""RD_SOLVER_THOMAS solves a proposal on the interval by one algorithm whatever
batch it is in: results do not depend on the batch, to the bit, and chains split
over objects reproduce one object's at any number of chains."""
import numpy as np
import pytest
import torch

import paper_1605_04718_gb300 as rd
import rd_synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
BIG = 21000  # above the count from which a thread per proposal is the default


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1605_04718_gb300 import build
    build.build()
    rd.load()


def _problem(n, steps, growth=False):
    rng = np.random.default_rng(n)
    w0 = np.array([1.0, 0.9])[:, None] + rng.uniform(-0.05, 0.05, (2, n))
    y = w0[None] + rng.normal(0, 0.02, (1, 2, n))
    pm = [0, 1, 2, 4] if growth else [0, 1, 2]
    desc = rd.make_desc(1, [n], 1e-4, steps, pm, [0.1, 0.9, 10.0, 200.0, 0.0],
                        [rd.RD_PRIOR_UNIFORM] * len(pm), [0.0] * len(pm), [100.0] * len(pm),
                        [rd.RD_STEP_LINEAR] * len(pm), growth=1 if growth else 0,
                        solver=rd.RD_SOLVER_THOMAS)
    p = rd.rd_problem_create(desc)
    rd.rd_set_initial_state(p, 0, w0[0], w0[1])
    rd.rd_set_observations(p, 0, [steps], 3, y, 0.02)
    return p


def _eval(p, theta, n):
    B = len(theta)
    th = torch.tensor(theta, dtype=torch.float64, device=DEV)
    phi = torch.zeros(B, dtype=torch.float64, device=DEV)
    st = torch.zeros(B, dtype=torch.int32, device=DEV)
    fl = torch.zeros((B, 2, n), dtype=torch.float64, device=DEV)
    rd.rd_evaluate_batch(p, th, phi, st, fields=fl)
    rd.rd_sync(p)
    return phi.cpu().numpy(), st.cpu().numpy(), fl.cpu().numpy()


def _theta(batch):
    return rd_synth.lognormal_draws([0.1, 0.9, 10.0], [0.1] * 3, batch, seed=batch)


@pytest.mark.parametrize("n", [20, 64, 100])
@pytest.mark.parametrize("growth", [False, True])
def test_results_do_not_depend_on_the_batch(n, growth):
    p = _problem(n, 20, growth)
    big = _theta(BIG)
    if growth:
        big = np.column_stack([big, np.linspace(0.0, 0.05, BIG)])
    ref = _eval(p, big, n)
    for batch in (1, 5, 700):
        for a, b in zip(_eval(p, big[:batch], n), ref):
            assert np.array_equal(a, b[:batch]), batch
    rd.rd_problem_destroy(p)


def test_small_objects_reproduce_the_chains_of_a_large_one():
    p = _problem(24, 20)
    theta0 = _theta(BIG)

    def run(first, count):
        c = rd.rd_chains_create(p, theta0[first:first + count], 5, [0.01] * 3, capacity=3)
        if first:
            rd.rd_chains_set_first_chain(c, first)
        rd.rd_chains_run(c, 3)
        s, _ = rd.rd_chains_read_samples(c, 3, 3, count)
        _, phi = rd.rd_chains_get_state(c, 3, count)
        rd.rd_chains_destroy(c)
        return s, phi

    whole, phi = run(0, BIG)
    for first, count in ((0, 9), (12345, 50)):
        s, f = run(first, count)
        assert np.array_equal(s, whole[..., first:first + count])
        assert np.array_equal(f, phi[first:first + count])
    rd.rd_problem_destroy(p)
