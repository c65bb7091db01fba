"""The interval's solve kernel spreads a proposal over one warp, over 8 lanes or
gives it one thread, by the size of the batch: every path against the FP64
oracle at grid sizes around the lanes' node counts, and the semi-implicit step
the same to the bit on all of them."""
import numpy as np
import pytest
import torch

import oracle
import paper_1605_04718_gb300 as rd
import rd_synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
TRUE3 = [0.1, 0.9, 10.0]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1605_04718_gb300 import build
    build.build()
    oracle.build()
    rd.load()


def _problem(n, steps, scheme, growth):
    rng = np.random.default_rng(n)
    w0 = np.array([1.0, 0.9])[:, None] + rng.uniform(-0.05, 0.05, (2, n))
    marks = [2, steps]
    y = w0[None] + rng.normal(0, 0.02, (2, 2, n))
    pm = [0, 1, 2, 4] if growth else [0, 1, 2]
    desc = rd.make_desc(1, [n], 1e-4, steps, pm, [0.1, 0.9, 10.0, 200.0, 0.0],
                        [rd.RD_PRIOR_UNIFORM] * len(pm), [0.0] * len(pm), [100.0] * len(pm),
                        [rd.RD_STEP_LINEAR] * len(pm), growth=1 if growth else 0)
    p = rd.rd_problem_create(desc)
    rd.rd_set_initial_state(p, 0, w0[0], w0[1])
    rd.rd_set_observations(p, 0, marks, 3, y, 0.02)
    if scheme == "picard":
        rd.rd_set_scheme(p, rd.RD_SCHEME_PICARD)
    P = oracle.Problem(1, n, 1e-4, steps, w0[0], w0[1], y=y, obs_steps=marks, field_mask=3,
                       sigma=0.02, scheme=scheme)
    return p, P


def _eval(p, theta, n):
    B = len(theta)
    th = torch.tensor(theta, dtype=torch.float64, device=DEV)
    phi = torch.zeros(B, dtype=torch.float64, device=DEV)
    st = torch.zeros(B, dtype=torch.int32, device=DEV)
    fl = torch.zeros((B, 2, n), dtype=torch.float64, device=DEV)
    rd.rd_evaluate_batch(p, th, phi, st, fields=fl)
    rd.rd_sync(p)
    return phi.cpu().numpy(), st.cpu().numpy(), fl.cpu().numpy()


def _theta(batch, growth):
    t = rd_synth.lognormal_draws(TRUE3, [0.1] * 3, batch, seed=batch)
    return np.column_stack([t, np.linspace(0.0, 0.05, batch)]) if growth else t


@pytest.mark.parametrize("n", [2, 3, 15, 16, 17, 33, 64, 65, 100, 129, 200, 256])
@pytest.mark.parametrize("growth", [False, True])
@pytest.mark.parametrize("batch", [3, 21000])
def test_imex_paths_match_the_oracle(n, growth, batch):
    """Fields to 1e-12 after 5 steps (FP64 rounding, at most some hundred units
    in the last place per step, of solutions of order 1)."""
    if batch > 3 and n > 100:
        pytest.skip("one thread per proposal is covered by the smaller grids")
    p, P = _problem(n, 5, "imex", growth)
    theta = _theta(batch, growth)
    theta[1, 2] = 0.0  # no diffusion of v
    phi, st, fl = _eval(p, theta, n)
    rd.rd_problem_destroy(p)
    for i in (0, 1, batch - 1):
        full = [theta[i, 0], theta[i, 1], theta[i, 2], 200.0, theta[i, 3] if growth else 0.0]
        po, so, uo, vo = P.forward(full)
        assert st[i] == so == 0
        assert np.abs(fl[i] - np.stack([uo, vo])).max() < 1e-12, i
        assert abs(phi[i] - po) <= 1e-9 * po


def test_negative_diffusion_is_still_eliminated():
    p, P = _problem(20, 5, "imex", False)
    theta = _theta(5, False)
    theta[2, 2] = -0.01
    phi, st, fl = _eval(p, theta, 20)
    rd.rd_problem_destroy(p)
    for i in range(5):
        po, so, uo, vo = P.forward([*theta[i], 200.0, 0.0])
        assert st[i] == so == 0
        assert np.abs(fl[i] - np.stack([uo, vo])).max() < 1e-12, i


@pytest.mark.parametrize("n", [2, 31, 64, 100])
@pytest.mark.parametrize("growth", [False, True])
def test_semi_implicit_paths_agree_to_the_bit(n, growth):
    p, P = _problem(n, 5, "picard", growth)
    big = _theta(30000, growth)
    ref = _eval(p, big, n)  # one thread per proposal
    for batch in (1, 3, 1301):  # a warp each, a warp each, 8 lanes each
        got = _eval(p, big[:batch], n)
        for a, b in zip(got, ref):
            assert np.array_equal(a, b[:batch]), batch
    rd.rd_problem_destroy(p)
    po, so, uo, vo = P.forward([big[0, 0], big[0, 1], big[0, 2], 200.0, 0.0])
    if not growth:
        assert np.abs(ref[2][0] - np.stack([uo, vo])).max() < 1e-12
