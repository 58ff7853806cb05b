"""Timing cases of the sampler's public entry points.

Each case is one call a sampling program makes: a chain (`hmc_sample_chain`,
its streaming form, or `Sampler.sample_chain`) of one posterior family, or
the batched log-density with its gradient through the autograd binding.  The
targets and sizes are those of `paper_2002_01184_gb300.workloads` (the worked
example, the correlated Gaussian, the logistic regression, the funnels and
the uneven batch's ranges) with shorter chains.

A chain's starting state, data and step size come from the case's seed; a
pass restarts the chain at the same state.  Past its first few transitions a
chain in float64 is another chain (one accept decision that falls the other
way changes the rest of that chain), so only the gradient cases have a
float64 value.
"""
import math

import torch

from paper_2002_01184_gb300 import autograd, hmc, workloads
from paper_2002_01184_gb300.sampler import Sampler


def listed():
    return [
        # the worked example of the paper's introduction: 100 chains of one
        # dimension, through the convenience class: the smallest call
        {"name": "worked_example", "call": "sampler", "kind": "std_normal", "chains": 100, "dim": 1,
         "rows": 0, "steps": 3, "eps": 1.5, "burnin": 300, "kept": 100, "adapt": False},
        # a hierarchical posterior (Neal's funnel), many chains, adapting
        {"name": "funnel_chain", "call": "chain", "kind": "funnel", "chains": 4096, "dim": 100,
         "rows": 0, "steps": 10, "eps": 0.1, "burnin": 50, "kept": 100, "adapt": True},
        # the dense Gaussian at the benchmark's size
        {"name": "gauss_chain", "call": "chain", "kind": "corr_gauss", "chains": 4096, "dim": 256,
         "rows": 0, "steps": 16, "eps": 0.0625, "burnin": 20, "kept": 40, "adapt": True},
        # a smaller dense Gaussian without a trace: running moments and
        # batch-means effective sample sizes instead
        {"name": "gauss_streaming", "call": "streaming", "kind": "corr_gauss", "chains": 1000, "dim": 100,
         "rows": 0, "steps": 16, "eps": 0.1, "burnin": 20, "kept": 40, "adapt": True},
        # a dense Gaussian wider than the benchmark's
        {"name": "gauss_wide", "call": "chain", "kind": "corr_gauss", "chains": 2048, "dim": 512,
         "rows": 0, "steps": 16, "eps": 0.044, "burnin": 10, "kept": 10, "adapt": True},
        # Bayesian logistic regression at the benchmark's size: the largest
        {"name": "logreg_chain", "call": "chain", "kind": "logreg", "chains": 2048, "dim": 128,
         "rows": 20000, "steps": 10, "eps": 0.0088, "burnin": 5, "kept": 10, "adapt": True},
        # ... with more features than one tensor-core tile is wide, ragged
        {"name": "logreg_wide", "call": "chain", "kind": "logreg", "chains": 700, "dim": 301,
         "rows": 8000, "steps": 10, "eps": 0.0058, "burnin": 5, "kept": 10, "adapt": True},
        # ... and a small data set, as most posteriors of a batch or a server
        {"name": "logreg_small", "call": "chain", "kind": "logreg", "chains": 64, "dim": 11,
         "rows": 800, "steps": 10, "eps": 0.03, "burnin": 50, "kept": 50, "adapt": True},
        # the No-U-Turn Sampler, dense Gaussian, step size as adapted
        {"name": "nuts_gauss", "call": "nuts", "kind": "corr_gauss", "chains": 4096, "dim": 256,
         "rows": 0, "steps": 10, "eps": 0.4, "burnin": 0, "kept": 10, "adapt": False},
        # ... on the funnel, whose trees differ most from chain to chain
        {"name": "nuts_funnel", "call": "nuts", "kind": "funnel", "chains": 1024, "dim": 100,
         "rows": 0, "steps": 10, "eps": 0.175, "burnin": 0, "kept": 20, "adapt": False},
        # random-walk Metropolis-Hastings: one density evaluation a transition
        {"name": "random_walk", "call": "random_walk", "kind": "corr_gauss", "chains": 4096, "dim": 256,
         "rows": 0, "steps": 1, "eps": 0.1, "burnin": 10, "kept": 20, "adapt": True},
        # log p and its gradient through torch.autograd, as a variational fit
        # or an optimiser uses the target
        {"name": "logreg_autograd", "call": "autograd", "kind": "logreg", "chains": 2048, "dim": 128,
         "rows": 20000, "steps": 1, "eps": 0.0, "burnin": 0, "kept": 0, "adapt": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    """A case of the same families, sizes spread over the workloads' ranges."""
    call = rng.choice(["sampler", "chain", "chain", "chain", "streaming", "nuts", "random_walk", "autograd"])
    if call == "sampler":
        kind = "std_normal"
    elif call in ("nuts", "random_walk"):
        kind = rng.choice(["corr_gauss", "funnel"])
    elif call == "streaming":
        kind = rng.choice(["corr_gauss", "funnel"])
    elif call == "autograd":
        kind = rng.choice(["corr_gauss", "logreg"])
    else:
        kind = rng.choice(["funnel", "corr_gauss", "logreg"])
    chains = _log_int(rng, 64, 4096)
    rows, steps, burnin, kept, adapt = 0, 10, 10, 20, True
    if kind == "std_normal":
        dim = _log_int(rng, 1, 128)
        steps, burnin, kept, adapt = rng.randint(1, 8), rng.randint(0, 300), rng.randint(50, 300), False
        eps = 1.5 / dim ** 0.25
    elif kind == "funnel":
        dim = rng.randint(10, 200)
        eps = 0.1
        burnin, kept = rng.randint(10, 60), rng.randint(20, 100)
    elif kind == "corr_gauss":
        dim = 4 * _log_int(rng, 8, 128)
        if rng.random() < 0.2:       # every dimension is taken, odd ones too
            dim -= rng.randint(1, 3)
        if dim > 256:
            chains = _log_int(rng, 64, 2048)
        steps = 16
        eps = 1.0 / math.sqrt(dim)
        burnin, kept = rng.randint(5, 10), rng.randint(10, 20)
    else:
        while True:
            dim, rows = _log_int(rng, 8, 512), _log_int(rng, 500, 20000)
            if dim > 128 and chains * dim * rows > 700 * 301 * 8000 or \
                    chains * dim * rows > 2048 * 128 * 20000:
                chains = max(64, chains // 2)
                continue
            break
        eps = 0.1 / math.sqrt(dim)
        burnin, kept = 5, 10
    if call == "nuts":
        adapt, steps, burnin = False, 10, 0
        if kind == "corr_gauss":
            dim = min(256, (dim + 3) // 4 * 4)     # the sampler wants multiples of 4
            kept, eps = rng.randint(4, 10), 0.4
        else:
            kept, eps = rng.randint(8, 20), 0.175
            chains = min(chains, 1024)
    elif call == "random_walk":
        steps, eps = 1, 1.6 / math.sqrt(dim)
    elif call == "autograd":
        steps, burnin, kept, adapt, eps = 1, 0, 0, False, 0.0
    return {"call": call, "kind": kind, "chains": chains, "dim": dim, "rows": rows, "steps": steps,
            "eps": eps, "burnin": burnin, "kept": kept, "adapt": adapt}


def _inputs(case, seed):
    """Target data and starting state on the GPU, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    C, D, N = case["chains"], case["dim"], case["rows"]
    kw = {"device": "cuda", "generator": gen}
    data = {}
    if case["kind"] == "corr_gauss":
        A = torch.randn(D, D, dtype=torch.float64, **kw)
        P = (A @ A.T / D + 0.1 * torch.eye(D, dtype=torch.float64, device="cuda")).float()
        data["P"] = 0.5 * (P + P.T)
    elif case["kind"] == "logreg":
        data["X"] = torch.randn(N, D, **kw)
        w = torch.randn(D, **kw) / math.sqrt(D)
        data["y"] = (torch.rand(N, **kw) < torch.sigmoid(data["X"] @ w)).float()
    x0 = torch.randn(C, D, **kw)
    if case["kind"] == "std_normal":
        x0.mul_(0.1)
    if case["kind"] == "logreg":
        x0.mul_(1.0 / math.sqrt(D))
    return data, x0, gen


def prepare(case, seed):
    data, x0, gen = _inputs(case, seed)
    C, D, K = case["chains"], case["dim"], case["kept"]
    state = {"case": case, "x0": x0}
    if case["call"] == "autograd":
        state["target"] = autograd.Target(case["kind"], D, **data)
        state["weights"] = torch.rand(C, device="cuda", generator=gen) + 0.5
        return state
    proposal = {"nuts": hmc.HMC_PROPOSAL_NUTS,
                "random_walk": hmc.HMC_PROPOSAL_RANDOM_WALK}.get(case["call"], hmc.HMC_PROPOSAL_LEAPFROG)
    problem = workloads.Problem(
        case["kind"], D, C, None, num_leapfrog=case["steps"], step_size=case["eps"], adapt=case["adapt"],
        target_accept=0.8 if case["kind"] in ("logreg", "funnel") else 0.65,
        num_burnin=case["burnin"], num_results=K, seed=seed, **data)
    state["sampler"] = Sampler(problem, proposal=proposal)
    state["x"] = torch.empty_like(x0)
    if case["call"] == "sampler":
        return state
    state["eps"] = torch.empty(K, device="cuda")
    state["accepted"] = torch.empty(K, C, dtype=torch.uint8, device="cuda")
    if case["call"] == "streaming":
        state["mean"], state["m2"] = torch.empty_like(x0), torch.empty_like(x0)
        state["ess"] = torch.empty(D, device="cuda")
    else:
        state["samples"] = torch.empty(K, C, D, device="cuda")
    return state


def run(state):
    case = state["case"]
    if case["call"] == "autograd":
        x = state["x0"].detach().requires_grad_(True)
        lp = autograd.log_prob(x, state["target"])
        (dx,) = torch.autograd.grad(lp, x, state["weights"])
        return {"log_prob": lp.detach(), "dx": dx}
    s, x, B, K = state["sampler"], state["x"], case["burnin"], case["kept"]
    x.copy_(state["x0"])
    if case["call"] == "sampler":
        samples, eps, accepted = s.sample_chain(x, B, K)
        return {"x": x, "samples": samples, "eps": eps, "accepted": accepted}
    if case["call"] == "streaming":
        hmc.hmc_sample_chain_streaming_ess(s.ctx, x, B, K, max(1, K // 4), state["mean"], state["m2"],
                                           state["ess"], state["eps"], state["accepted"])
        return {k: state[k] for k in ("x", "mean", "m2", "ess", "eps", "accepted")}
    hmc.hmc_sample_chain(s.ctx, x, B, K, state["samples"], state["eps"], state["accepted"])
    return {k: state[k] for k in ("x", "samples", "eps", "accepted")}


def work(case):
    C, D, N, L = case["chains"], case["dim"], case["rows"], case["steps"]
    T, K = case["burnin"] + case["kept"], case["kept"]
    grad = {"std_normal": 4.0 * D, "funnel": 8.0 * D, "corr_gauss": 2.0 * D * D,
            "logreg": 4.0 * N * D}[case["kind"]]
    data = {"corr_gauss": 4.0 * D * D, "logreg": 4.0 * N * (D + 1)}.get(case["kind"], 0.0)
    if case["call"] == "autograd":
        # forward and backward are calls of their own: each evaluates both products
        return {"bytes": 2 * data + 4.0 * C * (3 * D + 2), "flops": 2 * C * grad}
    if case["call"] == "nuts":
        # leapfrog steps of a tree depend on the chain: the mean tree of these
        # step sizes (about 24 leaves on the Gaussian, 67 on the funnel)
        L = 24 if case["kind"] == "corr_gauss" else 67
    evals = C * (1.0 + T * (1 if case["call"] == "random_walk" else L))
    out = 4.0 * D + 4.0 * D if case["call"] == "streaming" else 4.0 * K * D
    return {"bytes": data + C * (8.0 * D + out + K), "flops": evals * (grad + 6.0 * D)}


def exact(case, seed):
    if case["call"] != "autograd":
        return None
    data, x0, gen = _inputs(case, seed)
    weights = (torch.rand(case["chains"], device="cuda", generator=gen) + 0.5).double()
    x = x0.double()
    if case["kind"] == "corr_gauss":
        g = -(x @ data["P"].double())
        lp = 0.5 * (x * g).sum(1)
    else:
        X, y = data["X"].double(), data["y"].double()
        z = x @ X.T
        lp = (z * y - torch.nn.functional.softplus(z, threshold=1e9)).sum(1) - 0.5 * x.square().sum(1)
        g = (y - torch.sigmoid(z)) @ X - x
    return {"log_prob": lp, "dx": weights[:, None] * g}
