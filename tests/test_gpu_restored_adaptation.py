"""A restored adaptation state decides which transitions still adapt, also where
the context that takes it was created with another schedule: the launches that run
many transitions go by the state, as single transitions do."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402


@pytest.mark.parametrize("kind,nuts", [("std_normal", False), ("funnel", False), ("logreg", False), ("corr_gauss", False),
                                       ("funnel", True)])
@pytest.mark.parametrize("adapt_steps", [None, 7, 30])
def test_restored_schedule_is_the_saved_one(kind, nuts, adapt_steps):
    C, D, N, saved_steps, k, n = 96, 8, 200, 12, 5, 20
    gen = torch.Generator(device="cuda").manual_seed(1)
    data = {}
    if kind == "logreg":
        data = {"X": torch.randn(N, D, device="cuda", generator=gen),
                "y": (torch.rand(N, device="cuda", generator=gen) < 0.5).float()}
    if kind == "corr_gauss":
        data = {"P": torch.eye(D, device="cuda")}
    target = H.make_target(kind, D, **data)
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    kw = {"seed": 3, "target_accept": 0.8,
          "proposal": H.HMC_PROPOSAL_NUTS if nuts else H.HMC_PROPOSAL_LEAPFROG}
    first = H.hmc_create(target, C, H.make_config(4, 0.1, adapt=True, num_adapt_steps=saved_steps, **kw))
    x = x0.clone()
    H.hmc_sample_chain_range(first, x, 0, 0, k)
    state, xk = H.hmc_save_state(first), x.clone()
    ref = torch.empty(n - k, C, D, device="cuda")
    H.hmc_sample_chain_range(first, x, 0, k, n, ref)
    H.hmc_synchronize(first)
    second = H.hmc_create(target, C, H.make_config(4, 0.1, adapt=adapt_steps is not None,
                                                   num_adapt_steps=adapt_steps or 0, **kw))
    H.hmc_restore_state(second, state)
    y, got = xk.clone(), torch.empty_like(ref)
    H.hmc_sample_chain_range(second, y, 0, k, n, got)
    H.hmc_synchronize(second)
    assert torch.equal(got, ref) and torch.equal(y, x)
    assert H.hmc_read_adaptation(second) == H.hmc_read_adaptation(first)
    H.hmc_destroy(first)
    H.hmc_destroy(second)
