"""Calls that take one of two launch forms by their size: the results do not
depend on it.  Sizes on both sides of the lines."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import numpy as np  # noqa: E402

from paper_2002_01184_gb300 import hmc as H  # noqa: E402
from tests.test_gpu_chain_launch import chain, check_equal  # noqa: E402


# one transition per call (tiles for many chains of more than 64 dims) against
# the whole chain in one launch
@pytest.mark.parametrize("kind,C,D,L", [("std_normal", 3000, 100, 1), ("std_normal", 2400, 100, 9), ("funnel", 2600, 65, 7),
                                        ("funnel", 2600, 65, 8), ("std_normal", 1217, 129, 3), ("funnel", 1216, 300, 2),
                                        ("funnel", 1300, 260, 2), ("std_normal", 1500, 513, 2), ("funnel", 1250, 1023, 1)])
@pytest.mark.parametrize("adapt", [False, True])
def test_single_transitions_equal_the_chain(kind, C, D, L, adapt):
    gen = torch.Generator(device="cuda").manual_seed(C + D)
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    B, K = 3, 3
    cfg = H.make_config(L, 0.4 / D ** 0.25, seed=7, adapt=adapt, target_accept=0.8, num_adapt_steps=B, chain_offset=5)
    x, s, e, a, da = chain(H.make_target(kind, D), cfg, x0, B, K, False)
    ctx = H.hmc_create(H.make_target(kind, D), C, cfg)
    y = x0.clone()
    H.hmc_bootstrap(ctx, y)
    for t in range(B + K):
        H.hmc_step(ctx, y, t)
        if t >= B:
            assert torch.equal(y, s[t - B])
    H.hmc_synchronize(ctx)
    assert H.hmc_read_adaptation(ctx) == da
    H.hmc_destroy(ctx)


def logreg(N, D, C):
    gen = torch.Generator(device="cuda").manual_seed(N * 10007 + C)
    X = torch.randn(N, D, device="cuda", generator=gen)
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    return X, y, torch.randn(C, D, device="cuda", generator=gen) / D ** 0.5


# few rows and many chains: tiles, a launch per transition; some of these sizes take
# them for single transitions only, or while the step size adapts
LOGREG = [(17, 4, 2400, 1), (17, 4, 2400, 10), (17, 4, 9000, 3), (100, 4, 5000, 1), (64, 20, 3000, 2), (30, 60, 5000, 2),
          (200, 4, 2400, 1)]


@pytest.mark.parametrize("N,D,C,L", LOGREG)
@pytest.mark.parametrize("adapt,B,K", [(False, 2, 5), (True, 5, 3)])
def test_small_logreg_with_many_chains(N, D, C, L, adapt, B, K):
    X, y, x0 = logreg(N, D, C)
    cfg = H.make_config(L, 0.5 / (N * D) ** 0.5, seed=11, adapt=adapt, target_accept=0.8, num_adapt_steps=B,
                        impl=H.HMC_IMPL_FUSED_SIMT)
    target = H.make_target("logreg", D, X=X, y=y)
    if N * D * C <= 1 << 22:          # what a batch groups
        check_equal(target, cfg, x0, B, K)
    x, s, e, a, da = chain(target, cfg, x0, B, K, False)
    ctx = H.hmc_create(target, C, cfg)
    y1 = x0.clone()
    H.hmc_bootstrap(ctx, y1)
    for t in range(B + K):
        H.hmc_step(ctx, y1, t)
        assert t < B or torch.equal(y1, s[t - B])
    H.hmc_synchronize(ctx)
    assert H.hmc_read_adaptation(ctx) == da
    H.hmc_destroy(ctx)


@pytest.mark.parametrize("N,D,C,L", LOGREG[:4])
@pytest.mark.parametrize("adapt_steps", [0, 4, 12])
def test_small_logreg_with_many_chains_streams_its_moments(N, D, C, L, adapt_steps):
    X, y, x0 = logreg(N, D, C)
    B, K = 4, 8                     # (12 adapting transitions: some kept ones adapt)
    cfg = H.make_config(L, 0.5 / (N * D) ** 0.5, seed=11, adapt=adapt_steps > 0, target_accept=0.8,
                        num_adapt_steps=adapt_steps, impl=H.HMC_IMPL_FUSED_SIMT)
    target = H.make_target("logreg", D, X=X, y=y)
    x, s, _, _, da = chain(target, cfg, x0, B, K, False)
    ctx = H.hmc_create(target, C, cfg)
    x2 = x0.clone()
    mean, m2, ess = torch.empty_like(x2), torch.empty_like(x2), torch.empty(D, device="cuda")
    H.hmc_sample_chain_streaming_ess(ctx, x2, B, K, 2, mean, m2, ess)
    H.hmc_synchronize(ctx)
    assert H.hmc_read_adaptation(ctx) == da
    H.hmc_destroy(ctx)
    assert torch.equal(x2, x)
    smp = s.double().cpu().numpy()
    scale = np.abs(smp).max(axis=0) + 1e-6
    # the tolerances of the streaming tests
    assert np.max(np.abs(mean.double().cpu().numpy() - smp.mean(axis=0)) / scale) < 1e-5
    ref_m2 = ((smp - smp.mean(axis=0)) ** 2).sum(axis=0)
    assert np.max(np.abs(m2.double().cpu().numpy() - ref_m2) / (scale ** 2 * K)) < 1e-5
    assert torch.isfinite(ess).all()


# NUTS on the Gaussian: a cluster per chain block or the grid-wide loop
@pytest.mark.parametrize("D,depth,sizes", [(64, 4, (10000, 4900, 40)), (128, 4, (5000, 90)), (128, 7, (5000, 90)),
                                           (160, 5, (5000, 200, 30)), (256, 6, (5000, 600, 300, 50))])
def test_nuts_chains_do_not_depend_on_the_loops_form(D, depth, sizes):
    gen = torch.Generator(device="cuda").manual_seed(D)
    A = torch.randn(D, D, device="cuda", generator=gen, dtype=torch.float64)
    P = (A @ A.T / D + 0.1 * torch.eye(D, device="cuda", dtype=torch.float64)).float().contiguous()
    x0 = torch.randn(max(sizes), D, device="cuda", generator=gen)
    target, first = H.make_target("corr_gauss", D, P=P), None
    for C in sizes:
        ctx = H.hmc_create(target, C, H.make_config(depth, 0.3, seed=9, proposal=H.HMC_PROPOSAL_NUTS))
        x, s = x0[:C].clone(), torch.empty(3, C, D, device="cuda")
        a = torch.empty(3, C, dtype=torch.uint8, device="cuda")
        H.hmc_sample_chain(ctx, x, 1, 3, s, None, a)
        H.hmc_synchronize(ctx)
        H.hmc_destroy(ctx)
        if first is None:
            first = s, a
        assert torch.equal(s, first[0][:, :C]) and torch.equal(a, first[1][:, :C])
    assert first[1].any()


# replica sets: tempered tiles against the chain launch's tempered form
@pytest.mark.parametrize("kind,D", [("std_normal", 100), ("funnel", 200)])
def test_replica_sets_do_not_depend_on_their_number(kind, D):
    betas = [1.0, 0.6, 0.3, 0.1]
    x0 = torch.randn(700 * 4, D, device="cuda", generator=torch.Generator(device="cuda").manual_seed(D))
    out = []
    for sets in (700, 20):
        ctx = H.hmc_remc_create(H.make_target(kind, D), sets, betas, H.make_config(3, 0.1, seed=13))
        x, s = x0[:4 * sets].clone(), torch.empty(4, 4 * sets, D, device="cuda")
        H.hmc_sample_chain(ctx, x, 2, 4, s)
        H.hmc_synchronize(ctx)
        H.hmc_destroy(ctx)
        out.append((x, s))
    assert torch.equal(out[0][0][:80], out[1][0]) and torch.equal(out[0][1][:, :80], out[1][1])
