"""The elementwise NUTS kernel's forms -- more registers for few chains, more
resident chains for many, span starts in shared memory or in scratch -- give
a chain the same draws: the first chains of a call that fills the device
against a call with these chains alone."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402


# one, two and four blocks of 128 dims per lane, their edges; depth 1 has no span
# starts, depth 10 at 500 dims keeps them in scratch
@pytest.mark.parametrize("kind", ["std_normal", "funnel"])
@pytest.mark.parametrize("D,depth", [(2, 1), (3, 10), (128, 6), (129, 5), (256, 3), (257, 5), (500, 10)])
def test_forms_agree(kind, D, depth):
    gen = torch.Generator(device="cuda").manual_seed(D)
    x0 = torch.randn(5000, D, device="cuda", generator=gen)
    out = []
    for C in (5000, 7):
        cfg = H.make_config(depth, 0.1, seed=11, proposal=H.HMC_PROPOSAL_NUTS)
        ctx = H.hmc_create(H.make_target(kind, D), C, cfg)
        x, s = x0[:C].clone(), torch.empty(4, C, D, device="cuda")
        e, a = torch.empty(4, device="cuda"), torch.empty(4, C, dtype=torch.uint8, device="cuda")
        H.hmc_sample_chain(ctx, x, 1, 4, s, e, a)
        H.hmc_synchronize(ctx)
        H.hmc_destroy(ctx)
        out.append((x[:7], s[:, :7], a[:, :7]))
    for u, v in zip(*out):
        assert torch.equal(u, v)
    assert out[1][2].any()
