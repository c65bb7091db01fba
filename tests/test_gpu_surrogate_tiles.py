"""The surrogate's row tiles: Phi~ does not depend on the batch a row is in, at
batch sizes around the tile edges, and the gradient of a batch is the mean of
its parts', at batches of one tile, of more tiles than row shares, and between."""
import numpy as np
import pytest
import torch

import paper_1605_04718_gb300 as rd
import rd_synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0") if torch.cuda.is_available() else None
TRUE4 = [0.1, 0.9, 10.0, 200.0]


@pytest.fixture(scope="module")
def net():
    from paper_1605_04718_gb300 import build
    build.build()
    rd.load()
    desc = rd.make_desc(2, [32], 2.5e-4, 10, [0, 1, 2, 3], TRUE4 + [0.0],
                        [rd.RD_PRIOR_LOGNORMAL] * 4, TRUE4, [0.5] * 4, [rd.RD_STEP_LOG] * 4)
    p = rd.rd_problem_create(desc)
    s = rd.rd_surrogate_create(p, 3)
    norm = np.concatenate([np.log(TRUE4), [0.0], [0.5] * 4, [1.0], [100.0, 3.0, 1.5]])
    rd.rd_surrogate_set_params(s, None, norm)
    yield s
    rd.rd_surrogate_destroy(s)
    rd.rd_problem_destroy(p)


def _theta(n, seed=0):
    t = rd_synth.lognormal_draws(TRUE4, [0.5] * 4, n, seed=seed)
    return torch.tensor(t, dtype=torch.float64, device=DEV)


def test_predict_is_the_same_in_every_batch(net):
    theta = _theta(20000)
    phi = torch.zeros(20000, dtype=torch.float64, device=DEV)
    rd.rd_surrogate_predict(net, theta, phi)
    for n in (1, 31, 32, 33, 127, 128, 129, 4096, 4865, 9729):
        part = torch.full((n,), -1.0, dtype=torch.float64, device=DEV)
        rd.rd_surrogate_predict(net, theta[:n].contiguous(), part)
        assert torch.equal(part, phi[:n]), n


@pytest.mark.parametrize("tiles", [2, 5, 16, 17, 40])
def test_gradient_is_the_mean_over_tiles(net, tiles):
    B = 128 * tiles
    theta = _theta(B, seed=tiles)
    target = torch.randn(B, generator=torch.Generator().manual_seed(tiles)).to(DEV)
    n = rd.rd_surrogate_get_params(net)[0].size
    g = torch.zeros(n, dtype=torch.float32, device=DEV)
    loss = rd.rd_surrogate_loss_grad(net, theta, target, g)
    mean, acc = 0.0, torch.zeros(n, dtype=torch.float64, device=DEV)
    one = torch.zeros_like(g)
    for t in range(tiles):
        sl = slice(128 * t, 128 * (t + 1))
        mean += rd.rd_surrogate_loss_grad(net, theta[sl].contiguous(), target[sl].contiguous(), one)
        acc += one.double()
    assert abs(loss - mean / tiles) <= 1e-6 * loss
    # BF16 rounding of dZ acts on values scaled by 1 / B: relative 2^-9 per value at most
    acc /= tiles
    assert float((g.double() - acc).norm() / acc.norm()) < 2.0**-9
