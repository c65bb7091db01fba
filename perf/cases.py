"""Performance cases of the library: the calls its users make, each through the
public entry points, at sizes from the library's own workloads.

The library identifies the parameters of a reaction-diffusion system by MCMC,
so nearly all of a user's time is batched forward solves (``rd_evaluate_batch``
and the chains that call the same kernels); the rest is the surrogate network
of delayed-acceptance sampling.  Every case is a dict of plain values; ``kind``
says which calls it makes:

  solve2d    rd_evaluate_batch on FP32 fields, IMEX step (fixed or growing domain)
  host2d     the same solve called with host arrays, for a handful of proposals
  picard2d   the paper's semi-implicit step in 2-D
  chains1d   rd_chains_run on the FP64 interval: propose, solve, accept, read samples
  picard1d   the semi-implicit step on a growing interval (FP64)
  predict    the surrogate's forward pass
  grad       the surrogate's loss and gradient, one training batch

Horizons.  The stored 2-D workloads solve 8000 steps.  A step costs the same
whatever its index, but past the onset of the pattern two correct FP32 solves
drift apart (a rounding difference grows like the pattern itself, e-fold in
about 360 steps), so outputs could no longer be compared to FP32 accuracy.
The cases therefore stop at 100..1000 steps, with the whole batch of the
workload.  Phi of a 2-D solve is an FP64 sum over FP32 fields: it carries FP32
accuracy and is handed on as float32.
"""
import math

import numpy as np
import torch

import paper_1605_04718_gb300 as rd

TRUTH = (0.1, 0.9, 10.0, 200.0)  # a, b, d, gamma of every stored workload
GROWTH_RATE = 0.01
TAU_2D = 2.5e-4
E1_POLY = (0.6, 0.18, 0.036)  # exp(0.6 s) to third order: Example 1's exponential law
E1_RHO_T = math.exp(0.6)


# --------------------------------------------------------------------- cases
def listed():
    return [
        # One proposal after another from a host program (a sampler of the user's own, four
        # chains): host arrays in and out, the latency of a whole small call.
        dict(name="host_32", kind="host2d", sizes="32", batch=4, steps=100),
        # A coarse grid that is no power of two, a batch that is no multiple of anything.
        dict(name="solve_48", kind="solve2d", sizes="48", batch=777, steps=800, growth=0),
        # The 64^2 workload: 1024 chains in lock-step.
        dict(name="solve_64", kind="solve2d", sizes="64", batch=1024, steps=1000, growth=0),
        # The headline workload: 128^2, 4096 chains, one proposal each.
        dict(name="solve_128", kind="solve2d", sizes="128", batch=4096, steps=160, growth=0),
        # A few chains at 128^2 (a pilot run): fewer proposals than the chip has SMs.
        dict(name="few_128", kind="solve2d", sizes="128", batch=60, steps=1000, growth=0),
        # The growing-domain workload: matrices that change each step, u seen at five times.
        dict(name="grow_128", kind="solve2d", sizes="128", batch=608, steps=600, growth=1),
        # The uneven workload: a third each of 64^2, 96^2 and 128^2 in one call.
        dict(name="mixed", kind="solve2d", sizes="64+96+128", batch=1536, steps=400, growth=0),
        # The paper's semi-implicit step in 2-D, one proposal per SM.
        dict(name="picard_64", kind="picard2d", sizes="64", batch=152, steps=30),
        # The 1-D FP64 workload: 64 nodes, 4 chains, full horizon, two MCMC steps.
        dict(name="chains_1d", kind="chains1d", nodes=64, batch=4, steps=10000, mcmc=2),
        # Example 1: growth identification on 100 nodes, a batch of proposals.
        dict(name="example1_1d", kind="picard1d", nodes=100, batch=256, steps=1000),
        # Stage 1 of delayed acceptance: the surrogate on one proposal of each of 4096 chains.
        dict(name="predict", kind="predict", batch=4096),
        # One training batch of the surrogate: loss and all gradients.
        dict(name="grad", kind="grad", batch=1024),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve2d"] * 6 + ["host2d", "picard2d", "chains1d", "picard1d", "predict",
                                        "grad"])
    if kind == "solve2d":
        n_sizes = rng.choice([1, 1, 1, 2, 3])
        sizes = sorted(rng.sample([16, 32, 48, 64, 80, 96, 112, 128, 128], n_sizes))
        while len(set(sizes)) < n_sizes:
            sizes = sorted(rng.sample([16, 32, 48, 64, 80, 96, 112, 128], n_sizes))
        steps = spread(100, 1000)
        most = max(24, min(4096, int(4096 * 160 * 128 ** 3 / (steps * max(sizes) ** 3))))
        return dict(kind=kind, sizes="+".join(map(str, sizes)), batch=spread(20, most),
                    steps=steps, growth=int(rng.random() < 0.25))
    if kind == "host2d":
        return dict(kind=kind, sizes=str(16 * rng.randint(1, 8)), batch=rng.randint(1, 16),
                    steps=spread(50, 300))
    if kind == "picard2d":
        return dict(kind=kind, sizes=str(16 * rng.randint(2, 5)), batch=spread(20, 300),
                    steps=spread(8, 40))
    if kind == "chains1d":
        nodes = rng.randint(20, 200)
        return dict(kind=kind, nodes=nodes, batch=spread(2, 1500),
                    steps=spread(500, 400000 // nodes), mcmc=rng.randint(1, 2))
    if kind == "picard1d":
        nodes = rng.randint(32, 160)
        return dict(kind=kind, nodes=nodes, batch=spread(4, 1500), steps=spread(100, 80000 // nodes))
    if kind == "predict":
        return dict(kind=kind, batch=spread(64, 100000))
    return dict(kind=kind, batch=128 * spread(1, 64))


def _sizes(case):
    return [int(s) for s in case["sizes"].split("+")]


# -------------------------------------------------------------------- inputs
def _theta(rng, batch, centre, spread):
    """Parameter vectors of burned-in chains: about `spread` (relative) around the centre."""
    return np.asarray(centre) * np.exp(spread * rng.standard_normal((batch, len(centre))))


def _inputs_2d(case, seed):
    """Initial state and data of every size, parameters, size of every proposal: the stored
    workloads' recipe (steady state + U(-0.01, 0.01); data = a pattern about the steady state
    + N(0, 0.01^2)), float32 values."""
    rng = np.random.default_rng([seed, 2])
    batch, steps, growth = case["batch"], case["steps"], case.get("growth", 0)
    us, vs = TRUTH[0] + TRUTH[1], TRUTH[1] / (TRUTH[0] + TRUTH[1]) ** 2
    marks = [round(steps * o / 5) for o in range(1, 6)] if growth else [steps]
    sizes = []
    for n in _sizes(case):
        w0 = np.array([us, vs])[:, None, None] + rng.uniform(-0.01, 0.01, (2, n, n))
        x = np.cos(3 * math.pi * (np.arange(n) + 0.5) / n)
        base = np.array([us, vs])[:, None, None] + np.array([0.2, -0.1])[:, None, None] * np.outer(x, x)
        y = base[None, : 1 if growth else 2] + rng.normal(0, 0.01, (len(marks), 1 if growth else 2, n, n))
        sizes.append(dict(n=n, w0=w0.astype(np.float32).astype(np.float64),
                          y=y.astype(np.float32).astype(np.float64), marks=marks,
                          mask=1 if growth else 3, sigma=0.02 if growth else 0.01))
    theta = _theta(rng, batch, TRUTH, 0.002)
    if growth:
        theta = np.concatenate([theta, rng.uniform(0.0, 0.05, (batch, 1))], axis=1)
    which = np.arange(batch, dtype=np.int32) % len(sizes)
    return sizes, np.ascontiguousarray(theta), which, 1e-4 if growth else TAU_2D


def _inputs_1d(case, seed):
    rng = np.random.default_rng([seed, 1])
    n = case["nodes"]
    us, vs = TRUTH[0] + TRUTH[1], TRUTH[1] / (TRUTH[0] + TRUTH[1]) ** 2
    w0 = np.array([us, vs])[:, None] + rng.uniform(-0.01, 0.01, (2, n))
    return rng, w0


class Handles:
    """The library objects of one state, destroyed with it."""

    def __init__(self):
        self.problem = self.chains = self.surrogate = None

    def __del__(self):
        if self.chains is not None:
            rd.rd_chains_destroy(self.chains)
        if self.surrogate is not None:
            rd.rd_surrogate_destroy(self.surrogate)
        if self.problem is not None:
            rd.rd_problem_destroy(self.problem)


def prepare(case, seed):
    h = Handles()
    s = {"case": dict(case), "h": h}
    kind, dev = case["kind"], "cuda"
    if kind in ("solve2d", "host2d", "picard2d"):
        sizes, theta, which, tau = _inputs_2d(case, seed)
        g = case.get("growth", 0)
        p = 5 if g else 4
        desc = rd.make_desc(2, [z["n"] for z in sizes], tau, case["steps"], list(range(p)),
                            list(TRUTH) + [GROWTH_RATE if g else 0.0],
                            [rd.RD_PRIOR_LOGNORMAL] * 4 + [rd.RD_PRIOR_UNIFORM] * (p - 4),
                            list(TRUTH) + [0.0] * (p - 4), [0.5] * 4 + [0.05] * (p - 4),
                            [rd.RD_STEP_LOG] * 4 + [rd.RD_STEP_LINEAR] * (p - 4),
                            growth=rd.RD_GROWTH_EXP if g else rd.RD_GROWTH_NONE)
        h.problem = rd.rd_problem_create(desc)
        for k, z in enumerate(sizes):
            rd.rd_set_initial_state(h.problem, k, z["w0"][0], z["w0"][1])
            rd.rd_set_observations(h.problem, k, z["marks"], z["mask"], z["y"], z["sigma"])
        if kind == "picard2d":
            rd.rd_set_scheme(h.problem, rd.RD_SCHEME_PICARD)
        if kind == "host2d":
            s["theta"] = theta
            return s
        big, b = max(z["n"] for z in sizes), case["batch"]
        s["theta"] = torch.from_numpy(theta).to(dev)
        s["which"] = torch.from_numpy(which).to(dev) if len(sizes) > 1 else None
        s["phi"] = torch.zeros(b, dtype=torch.float64, device=dev)
        s["status"] = torch.zeros(b, dtype=torch.int32, device=dev)
        s["fields"] = torch.zeros((b, 2, big, big), dtype=torch.float32, device=dev)
    elif kind == "chains1d":
        rng, w0 = _inputs_1d(case, seed)
        y = _imex_1d(w0, np.array([TRUTH]), 1e-4, case["steps"])[0, 0]
        y = y + rng.normal(0, 0.01, y.shape)
        desc = rd.make_desc(1, [case["nodes"]], 1e-4, case["steps"], [0, 1], list(TRUTH) + [0.0],
                            [rd.RD_PRIOR_UNIFORM] * 2, [0.0, 0.0], [1.0, 2.0],
                            [rd.RD_STEP_LINEAR] * 2)
        h.problem = rd.rd_problem_create(desc)
        rd.rd_set_initial_state(h.problem, 0, w0[0], w0[1])
        rd.rd_set_observations(h.problem, 0, [case["steps"]], 1, y[None, None], 0.01)
        theta0 = _theta(rng, case["batch"], TRUTH[:2], 0.005)
        h.chains = rd.rd_chains_create(h.problem, theta0, seed, [0.01, 0.01], capacity=64)
    elif kind == "picard1d":
        rng, w0 = _inputs_1d(case, seed)
        y = (w0 + rng.normal(0, 0.05, w0.shape))[None]
        desc = rd.make_desc(1, [case["nodes"]], 1e-4, case["steps"], [5, 6, 7],
                            [0.1, 0.9, 10.0, 1000.0, 0.0] + list(E1_POLY),
                            [rd.RD_PRIOR_UNIFORM] * 3, [-2.0, -6.0, -6.0], [4.0, 6.0, 6.0],
                            [rd.RD_STEP_LINEAR] * 3, growth=rd.RD_GROWTH_POLY4, rho_T=E1_RHO_T)
        h.problem = rd.rd_problem_create(desc)
        rd.rd_set_initial_state(h.problem, 0, w0[0], w0[1])
        rd.rd_set_observations(h.problem, 0, [case["steps"]], 3, y, 0.05)
        rd.rd_set_scheme(h.problem, rd.RD_SCHEME_PICARD)
        b = case["batch"]
        s["theta"] = torch.from_numpy(_theta(rng, b, E1_POLY, 0.1)).to(dev)
        s["phi"] = torch.zeros(b, dtype=torch.float64, device=dev)
        s["status"] = torch.zeros(b, dtype=torch.int32, device=dev)
        s["fields"] = torch.zeros((b, 2, case["nodes"]), dtype=torch.float64, device=dev)
    else:
        params, norm, theta, target = _inputs_net(case, seed)
        desc = rd.make_desc(2, [128], TAU_2D, 8000, [0, 1, 2, 3], list(TRUTH) + [0.0],
                            [rd.RD_PRIOR_LOGNORMAL] * 4, list(TRUTH), [0.5] * 4,
                            [rd.RD_STEP_LOG] * 4)
        h.problem = rd.rd_problem_create(desc)
        h.surrogate = rd.rd_surrogate_create(h.problem, 0)
        rd.rd_surrogate_set_params(h.surrogate, params, norm)
        s["theta"] = torch.from_numpy(theta).to(dev)
        if kind == "predict":
            s["phi"] = torch.zeros(case["batch"], dtype=torch.float64, device=dev)
        else:
            s["target"] = torch.from_numpy(target).to(dev)
            s["grads"] = torch.zeros(params.size, dtype=torch.float32, device=dev)
    return s


# ----------------------------------------------------------------------- run
def run(s):
    case, h = s["case"], s["h"]
    kind = case["kind"]
    if kind in ("solve2d", "picard2d"):
        rd.rd_evaluate_batch(h.problem, s["theta"], s["phi"], s["status"], size_idx=s["which"],
                             fields=s["fields"])
        return {"fields": s["fields"], "phi": s["phi"].float(), "status": s["status"]}
    if kind == "host2d":
        phi, status = rd.rd_evaluate_batch_host(h.problem, s["theta"])
        return {"phi": phi.astype(np.float32), "status": status.astype(np.int64)}
    if kind == "chains1d":
        rd.rd_chains_run(h.chains, case["mcmc"])
        samples, counters = rd.rd_chains_read_samples(h.chains, case["mcmc"], 2, case["batch"])
        theta, phi = rd.rd_chains_get_state(h.chains, 2, case["batch"])
        return {"samples": samples, "counters": counters, "theta": theta, "phi": phi}
    if kind == "picard1d":
        rd.rd_evaluate_batch(h.problem, s["theta"], s["phi"], s["status"], fields=s["fields"])
        return {"fields": s["fields"], "phi": s["phi"], "status": s["status"]}
    if kind == "predict":  # Phi~ comes from an FP32-accumulating network: FP32 accuracy
        rd.rd_surrogate_predict(h.surrogate, s["theta"], s["phi"])
        return {"phi": s["phi"].float()}
    loss = rd.rd_surrogate_loss_grad(h.surrogate, s["theta"], s["target"], s["grads"])
    return {"loss": np.float32(loss), "grads": s["grads"]}


# ---------------------------------------------------------------------- work
def work(case):
    """Bytes: initial states, data and parameters in, outputs out.  Flops: per proposal and step
    of a 2-D solve the reaction (13 per point) and a direct solve of the two implicit systems
    (a fast transform each way in one direction, 2.5 log2 n per point, and a tridiagonal
    elimination, 5 per point, in the other); the semi-implicit step and the interval as written."""
    kind, b = case["kind"], case["batch"]
    if kind in ("solve2d", "host2d", "picard2d"):
        sizes = _sizes(case)
        per, io = 0.0, 0.0
        for n in sizes:
            per += n * n * (13 + 2 * (2 * 2.5 * math.log2(n) + 5)) * (3 if kind == "picard2d" else 1)
            io += n * n * 4 * 4
        out = 0 if kind == "host2d" else b * 2 * 4 * sum(n * n for n in sizes) / len(sizes)
        return {"bytes": io + out + b * (32 + 12), "flops": per / len(sizes) * b * case["steps"]}
    if kind == "chains1d":
        n = case["nodes"]
        return {"bytes": 24.0 * n + b * 16.0 * (2 * case["mcmc"] + 3),
                "flops": 22.0 * n * b * case["steps"] * case["mcmc"]}
    if kind == "picard1d":
        n = case["nodes"]
        return {"bytes": 32.0 * n + b * (24 + 12 + 16.0 * n), "flops": 40.0 * n * b * case["steps"]}
    w = rd.RD_SURROGATE_WIDTH
    mac = rd.SURROGATE_IN * w + 2 * w * w + w
    if kind == "predict":
        return {"bytes": 4.0 * (mac + 3 * w) + b * 40.0, "flops": 2.0 * mac * b}
    return {"bytes": 8.0 * (mac + 3 * w) + b * 36.0, "flops": 6.0 * mac * b}


# --------------------------------------------------------------------- exact
def _imex_2d(z, theta, tau, steps, growth, dev):
    """Fields at the observation steps and Phi in 64 bits: the IMEX step with the implicit solve
    in the cosine basis (even and odd halves apart, so each transform is two half-size products)."""
    n, h = z["n"], z["n"] // 2
    k = torch.arange(n, dtype=torch.float64, device=dev)[:, None]
    i = torch.arange(n, dtype=torch.float64, device=dev)[None]
    c = torch.cos(math.pi * k * (i + 0.5) / n) * math.sqrt(2 / n)
    c[0] = math.sqrt(1 / n)
    mu = 4 * torch.sin(math.pi * k[:, 0] / (2 * n)) ** 2
    ce, co, mu = c[0::2, :h].contiguous(), c[1::2, :h].contiguous(), torch.cat([mu[0::2], mu[1::2]])

    def fwd(x):  # last dimension -> even modes, then odd modes
        a, b = x[..., :h], x[..., h:].flip(-1)
        return torch.cat([(a + b) @ ce.T, (a - b) @ co.T], -1)

    def inv(x):
        a, b = x[..., :h] @ ce, x[..., h:] @ co
        return torch.cat([a + b, (a - b).flip(-1)], -1)

    a, b, d, g = [theta[:, j, None, None] for j in range(4)]
    r = theta[:, 4, None, None] if growth else torch.zeros_like(a)
    w0 = torch.from_numpy(z["w0"]).to(dev)
    y = torch.from_numpy(z["y"]).to(dev)
    u, v = w0[0].repeat(len(theta), 1, 1), w0[1].repeat(len(theta), 1, 1)
    lam = mu[:, None] + mu[None]
    phi = torch.zeros(len(theta), dtype=torch.float64, device=dev)
    diff = torch.stack([torch.ones_like(d), d], 1)
    den = None
    for s in range(1, steps + 1):
        u2v = u * u * v
        w = torch.stack([u + tau * g * (a - u + u2v), v + tau * g * (b - u2v)], 1)
        if growth or den is None:
            rho2 = torch.exp(2 * r * ((s - 1) * tau))[:, None]
            den = 1 + 2 * tau * r[:, None] + tau * n * n * diff / rho2 * lam
        w = fwd(fwd(w).transpose(-1, -2)) / den
        w = inv(inv(w).transpose(-1, -2))
        u, v = w[:, 0], w[:, 1]
        if s in z["marks"]:
            yo = y[z["marks"].index(s)]
            phi += ((yo - w[:, : yo.shape[0]]) ** 2).sum((1, 2, 3)) / (2 * z["sigma"] ** 2)
    return w, phi


def _exact_2d(case, seed, dev):
    sizes, theta, which, tau = _inputs_2d(case, seed)
    if sum(8.0 * z["n"] ** 3 for z in sizes) / len(sizes) * case["batch"] * case["steps"] > 1.4e13:
        return None
    big = max(z["n"] for z in sizes)
    fields = torch.zeros((case["batch"], 2, big * big), dtype=torch.float64)
    phi = torch.zeros(case["batch"], dtype=torch.float64)
    for k, z in enumerate(sizes):
        mine = np.nonzero(which == k)[0] if len(sizes) > 1 else np.arange(case["batch"])
        chunk = max(16, 60_000_000 // (2 * z["n"] ** 2 * 8))
        for lo in range(0, len(mine), chunk):
            at = mine[lo : lo + chunk]
            w, p = _imex_2d(z, torch.from_numpy(theta[at]).to(dev), tau, case["steps"],
                            case.get("growth", 0), dev)
            flat = fields.view(case["batch"], -1)
            flat[at, : 2 * z["n"] ** 2] = w.reshape(len(at), -1).cpu()
            phi[at] = p.cpu()
    status = None
    if case["kind"] == "host2d":
        return {"phi": phi, "status": status}
    return {"fields": fields.view(case["batch"], 2, big, big), "phi": phi, "status": status}


def _exact_picard_2d(case, seed, dev):
    """The semi-implicit step with conjugate gradients (diagonal scaling) to 1e-13."""
    (z,), theta, _, tau = _inputs_2d(case, seed)
    n = z["n"]
    th = torch.from_numpy(theta).to(dev)
    a, b, d, g = [th[:, j, None, None] for j in range(4)]
    w0, y = torch.from_numpy(z["w0"]).to(dev), torch.from_numpy(z["y"]).to(dev)
    u, v = w0[0].repeat(len(th), 1, 1), w0[1].repeat(len(th), 1, 1)

    def lap(x):
        p = torch.nn.functional.pad(x[:, None], (1, 1, 1, 1), mode="replicate")[:, 0]
        return p[:, 2:, 1:-1] + p[:, :-2, 1:-1] + p[:, 1:-1, 2:] + p[:, 1:-1, :-2] - 4 * x

    def dot(p, q):
        return (p * q).sum((1, 2), keepdim=True)

    def solve(diag, beta, rhs, x):
        m = 1 / (diag + 4 * beta)
        r = rhs - (diag * x - beta * lap(x))
        p = q = m * r
        rz, stop = dot(r, q), 1e-26 * dot(rhs, rhs)
        for it in range(400):
            ap = diag * p - beta * lap(p)
            al = rz / dot(p, ap)
            x, r = x + al * p, r - al * ap
            if it % 8 == 7 and bool((dot(r, r) <= stop).all()):
                break
            q = m * r
            new = dot(r, q)
            p, rz = q + new / rz * p, new
        return x

    for _ in range(case["steps"]):
        du, dv = 1 + tau * g * (1 - u * v), 1 + tau * g * u * u
        u, v = (solve(du, torch.full_like(a, tau * n * n), u + tau * g * a, u),
                solve(dv, tau * d * n * n, v + tau * g * b, v))
    w = torch.stack([u, v], 1)
    phi = ((y[0] - w) ** 2).sum((1, 2, 3)) / (2 * z["sigma"] ** 2)
    return {"fields": w, "phi": phi, "status": None}


def _imex_1d(w0, theta, tau, steps):
    """Final fields [B][2][n] on the interval: the inverse matrices applied as products."""
    n = w0.shape[1]
    lap = np.diag(np.full(n, -2.0)) + np.diag(np.ones(n - 1), 1) + np.diag(np.ones(n - 1), -1)
    lap[0, 0] = lap[-1, -1] = -1.0
    a, b, d, g = [theta[:, j, None] for j in range(4)]
    mu = np.linalg.inv(np.eye(n) - tau * n * n * lap)
    mv = np.linalg.inv(np.eye(n) - tau * float(d[0, 0]) * n * n * lap)  # one d for all
    u, v = np.repeat(w0[:1], len(theta), 0), np.repeat(w0[1:], len(theta), 0)
    for _ in range(steps):
        u2v = u * u * v
        u, v = (u + tau * g * (a - u + u2v)) @ mu, (v + tau * g * (b - u2v)) @ mv
    return np.stack([u, v], 1)


def _philox(chain, step, word, seed):
    """Philox4x32-10 (Salmon et al. 2011) of counters (chain, step, word, 0): 4 words each."""
    m = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, dtype=np.uint64) for x in (chain, np.full_like(chain, step),
                                                  np.full_like(chain, word), np.zeros_like(chain))]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for rnd in range(10):
        if rnd:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m]
    return c


def _exact_chains(case, seed):
    rng, w0 = _inputs_1d(case, seed)
    y = _imex_1d(w0, np.array([TRUTH]), 1e-4, case["steps"])[0, 0]
    y = y + rng.normal(0, 0.01, y.shape)
    theta = _theta(rng, case["batch"], TRUTH[:2], 0.005)

    def phi_of(t):
        full = np.concatenate([t, np.broadcast_to(TRUTH[2:], t.shape)], 1)
        u = _imex_1d(w0, full, 1e-4, case["steps"])[:, 0]
        return ((y - u) ** 2).sum(1) / (2 * 0.01 ** 2)

    phi = phi_of(theta)
    chain = np.arange(case["batch"], dtype=np.uint64)
    samples, tot = [], np.zeros(4)
    for step in range(case["mcmc"]):
        wd = _philox(chain, step, 0, seed) + _philox(chain, step, 1, seed)
        un = [(x.astype(np.float64) + 0.5) / 4294967296.0 for x in wd]
        rad, ang = np.sqrt(-2 * np.log(un[0])), 2 * math.pi * un[1]
        prop = theta + 0.01 * np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1)
        inside = ((prop >= 0) & (prop <= np.array([1.0, 2.0]))).all(1)
        pp = phi_of(np.where(inside[:, None], prop, theta))
        acc = inside & (np.log(un[6]) < phi - pp)
        theta, phi = np.where(acc[:, None], prop, theta), np.where(acc, pp, phi)
        samples.append(theta.T.copy())
        tot += [case["batch"], inside.sum(), acc.sum(), inside.sum()]
    return {"samples": np.stack(samples), "counters": tot, "theta": theta, "phi": phi}


def _exact_picard_1d(case, seed):
    """Example 1's step, every proposal's two systems eliminated at once."""
    rng, w0 = _inputs_1d(case, seed)
    y = w0 + rng.normal(0, 0.05, w0.shape)
    p = _theta(rng, case["batch"], E1_POLY, 0.1)
    n, steps, tau, b = case["nodes"], case["steps"], 1e-4, case["batch"]
    p1, p2, p3 = p.T
    p4 = E1_RHO_T - 1 - p1 - p2 - p3
    kin = np.array([0.1, 0.9])[:, None] * tau * 1000.0
    w = np.repeat(w0[:, None, :], b, 1).transpose(2, 0, 1).copy()  # [node][field][proposal]
    edge = np.full(n, 2.0)
    edge[0] = edge[-1] = 1.0
    for s in range(steps):
        t = s / steps
        rho = 1 + t * (p1 + t * (p2 + t * (p3 + t * p4)))
        q = (p1 + t * (2 * p2 + t * (3 * p3 + t * 4 * p4))) / (steps * tau) / rho
        beta = np.array([1.0, 10.0])[:, None] * tau * n * n / rho ** 2
        diag = np.stack([1 - w[:, 0] * w[:, 1], w[:, 0] ** 2], 1) * (tau * 1000.0) + 1 + tau * q
        diag += edge[:, None, None] * beta
        x = w + kin
        c = np.zeros_like(x)
        for i in range(n):
            den = diag[i] + (beta * c[i - 1] if i else 0.0)
            c[i] = -beta / den
            x[i] = (x[i] + (beta * x[i - 1] if i else 0.0)) / den
        for i in range(n - 2, -1, -1):
            x[i] -= c[i] * x[i + 1]
        w = x
    w = w.transpose(2, 1, 0)
    phi = ((y - w) ** 2).sum((1, 2)) / (2 * 0.05 ** 2)
    return {"fields": np.ascontiguousarray(w), "phi": phi, "status": None}


def _inputs_net(case, seed):
    """Weights as after training starts (He-uniform), the normalisation of a trained network,
    parameter vectors of the prior, standardised targets."""
    rng = np.random.default_rng([seed, 3])
    w, i = rd.RD_SURROGATE_WIDTH, rd.SURROGATE_IN
    w1 = rng.uniform(-1, 1, (w, i)) * math.sqrt(6 / 4)
    w1[:, 4:] = 0
    parts = [w1, 0.1 * rng.standard_normal(w)]
    for _ in range(2):
        parts += [rng.uniform(-1, 1, (w, w)) * math.sqrt(6 / w), 0.1 * rng.standard_normal(w)]
    parts += [rng.uniform(-1, 1, w) * 0.1 * math.sqrt(6 / w), np.zeros(1)]
    params = np.concatenate([x.ravel() for x in parts]).astype(np.float32)
    norm = np.concatenate([np.log(TRUTH), [0.0], [0.5] * 4, [1.0], [16000.0, 6.0, 1.5]])
    theta = _theta(rng, case["batch"], TRUTH, 0.5)
    return params, norm, theta, rng.standard_normal(case["batch"]).astype(np.float32)


def _exact_net(case, seed, dev):
    params, norm, theta, target = _inputs_net(case, seed)
    w, i = rd.RD_SURROGATE_WIDTH, rd.SURROGATE_IN
    flat = torch.from_numpy(params.astype(np.float64)).to(dev).requires_grad_(True)
    parts, at = [], 0
    for shape in ((w, i), (w,), (w, w), (w,), (w, w), (w,), (w,), (1,)):
        size = math.prod(shape)
        parts.append(flat[at : at + size].view(shape))
        at += size
    x = torch.zeros((case["batch"], i), dtype=torch.float64, device=dev)
    x[:, :4] = torch.from_numpy((np.log(theta) - norm[:4]) / norm[5:9]).to(dev)
    for k in range(3):
        x = torch.nn.functional.silu(x @ parts[2 * k].T + parts[2 * k + 1])
    out = x @ parts[6] + parts[7]
    if case["kind"] == "predict":
        return {"phi": (norm[10] + torch.exp(norm[11] + norm[12] * out)).detach()}
    loss = ((out - torch.from_numpy(target).to(dev).double()) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grads": flat.grad}


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind in ("solve2d", "host2d"):
        return _exact_2d(case, seed, dev)
    if kind == "picard2d":
        return _exact_picard_2d(case, seed, dev)
    if kind == "chains1d":
        return _exact_chains(case, seed)
    if kind == "picard1d":
        return _exact_picard_1d(case, seed)
    return _exact_net(case, seed, dev)
