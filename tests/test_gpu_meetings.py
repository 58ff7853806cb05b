"""Launches whose CTAs meet on the way: a meeting that cannot complete runs into
its time limit, the launch returns, the call reports it, and the next context
works.  The limit is a host-side setting; nothing faults or hangs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402


def gaussian(D):
    gen = torch.Generator(device="cuda").manual_seed(D)
    A = torch.randn(D, D, device="cuda", generator=gen, dtype=torch.float64)
    return (A @ A.T / D + 0.1 * torch.eye(D, device="cuda", dtype=torch.float64)).float().contiguous()


def run(target, cfg, x0, B, K):
    C, D = x0.shape
    ctx = H.hmc_create(target, C, cfg)
    x, s = x0.clone(), torch.empty(K, C, D, device="cuda")
    try:
        H.hmc_sample_chain(ctx, x, B, K, s)
        H.hmc_synchronize(ctx)
    finally:
        H.hmc_destroy(ctx)
    return x, s


def check_meeting_runs_out(target, cfg, x0, B, K, meeting, message):
    before = run(target, cfg, x0, B, K)
    try:
        H.hmc_debug_set_grid_barrier(20_000_000, meeting)
        with pytest.raises(H.HMCError) as err:
            run(target, cfg, x0, B, K)
        assert err.value.status == H.HMC_E_TIMEOUT and message in str(err.value)
    finally:
        H.hmc_debug_set_grid_barrier()
    after = run(target, cfg, x0, B, K)
    assert torch.equal(before[0], after[0]) and torch.equal(before[1], after[1])
    assert torch.isfinite(after[1]).all()


# one chain block and several; the meeting after the first step and the last one
@pytest.mark.parametrize("C,D,meeting", [(64, 260, 1), (300, 320, 3)])
def test_trajectory_launch(C, D, meeting):
    P = gaussian(D)
    x0 = torch.randn(C, D, device="cuda", generator=torch.Generator(device="cuda").manual_seed(C))
    cfg = H.make_config(4, 0.05, seed=5, use_graph=False)
    check_meeting_runs_out(H.make_target("corr_gauss", D, P=P), cfg, x0, 0, 1, meeting, "site 1")


# the dual-averaging meetings: CTA pairs, single CTAs
@pytest.mark.parametrize("C,D", [(128, 132), (4096, 256), (256, 128)])
@pytest.mark.parametrize("meeting", [1, 4])
def test_adapting_gaussian_chain(C, D, meeting):
    P = gaussian(D)
    x0 = torch.randn(C, D, device="cuda", generator=torch.Generator(device="cuda").manual_seed(C))
    cfg = H.make_config(3, 0.5 / D ** 0.5, seed=5, adapt=True, num_adapt_steps=4, use_graph=False)
    check_meeting_runs_out(H.make_target("corr_gauss", D, P=P), cfg, x0, 4, 2, meeting, "site 7")


# one CTA; CTAs of 8, 16 and 32 warps; chains that go through memory
@pytest.mark.parametrize("kind,C,D", [("std_normal", 5, 1), ("funnel", 300, 100), ("funnel", 1300, 100),
                                      ("funnel", 4096, 100), ("funnel", 9000, 100), ("funnel", 700, 1000)])
@pytest.mark.parametrize("meeting", [1, 4])
def test_adapting_elementwise_chain(kind, C, D, meeting):
    x0 = torch.randn(C, D, device="cuda", generator=torch.Generator(device="cuda").manual_seed(C))
    cfg = H.make_config(3, 0.1 / D ** 0.25, seed=5, adapt=True, num_adapt_steps=4, use_graph=False)
    check_meeting_runs_out(H.make_target(kind, D), cfg, x0, 4, 2, meeting, "grid barrier of a multi-transition launch")


# one chain; a group per CTA, four groups, several chains per group
@pytest.mark.parametrize("N,D,C", [(17, 3, 1), (800, 11, 64), (300, 8, 600), (100, 5, 2000)])
@pytest.mark.parametrize("meeting", [1, 4])
def test_adapting_logreg_chain(N, D, C, meeting):
    gen = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(N, D, device="cuda", generator=gen)
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    x0 = torch.randn(C, D, device="cuda", generator=gen) / D ** 0.5
    cfg = H.make_config(3, 0.3 / (N * D) ** 0.5, seed=5, adapt=True, num_adapt_steps=4, use_graph=False,
                        impl=H.HMC_IMPL_FUSED_SIMT)
    check_meeting_runs_out(H.make_target("logreg", D, X=X, y=y), cfg, x0, 4, 2, meeting,
                           "grid barrier of a multi-transition launch")


# 609 chains are 153 groups of four on 152 SMs, 9000 more elementwise chains than are
# resident: some CTAs have twice the work of others in every transition, which
# takes far longer here than a meeting may wait
@pytest.mark.parametrize("kind,N,D,C", [("logreg", 17, 2, 609), ("funnel", 0, 100, 9000)])
def test_long_transitions_do_not_run_into_the_limit(kind, N, D, C):
    gen = torch.Generator(device="cuda").manual_seed(C)
    data = {}
    if kind == "logreg":
        data = {"X": torch.randn(N, D, device="cuda", generator=gen),
                "y": (torch.rand(N, device="cuda", generator=gen) < 0.5).float()}
    target = H.make_target(kind, D, **data)
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    B, K = 2, 1
    cfg = H.make_config(20000, 1e-4, seed=5, adapt=True, num_adapt_steps=B, use_graph=False)
    try:
        H.hmc_debug_set_grid_barrier(1_000_000)
        x, s = run(target, cfg, x0, B, K)
    finally:
        H.hmc_debug_set_grid_barrier()
    ctx = H.hmc_create(target, C, cfg)
    y = x0.clone()
    H.hmc_bootstrap(ctx, y)
    for t in range(B + K):
        H.hmc_step(ctx, y, t)
    H.hmc_synchronize(ctx)
    H.hmc_destroy(ctx)
    assert torch.equal(x, y) and torch.equal(s[0], y)
