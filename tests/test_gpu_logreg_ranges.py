"""The tensor-core logistic regression's update over few and many ranges of data
rows: gradient and log p of the accepted states against float64."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402
from paper_2002_01184_gb300.sampler import device_view  # noqa: E402


# one range, a few, and as many as fill the SMs; one step and several
@pytest.mark.parametrize("C,N,D", [(300, 100, 8), (5000, 300, 30), (64, 900, 128), (64, 20000, 64)])
@pytest.mark.parametrize("L", [1, 3])
def test_update_against_float64(C, N, D, L):
    gen = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(N, D, device="cuda", generator=gen)
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    x = torch.randn(C, D, device="cuda", generator=gen) / D ** 0.5
    cfg = H.make_config(L, 0.05 / (N * D) ** 0.5, seed=3, impl=H.HMC_IMPL_FUSED_TENSOR)
    ctx = H.hmc_create(H.make_target("logreg", D, X=X, y=y), C, cfg)
    assert H.hmc_uses_tensor_cores(ctx)
    H.hmc_bootstrap(ctx, x)
    r = H.hmc_step(ctx, x, 0)
    H.hmc_synchronize(ctx)
    g = device_view(r.grad, (C, D), "<f4").clone().double()
    lp = device_view(r.target_log_prob, (C,), "<f4").clone().double()
    acc = device_view(r.is_accepted, (C,), "|u1").clone().bool()
    H.hmc_destroy(ctx)
    assert acc.float().mean() > 0.9
    x64, X64, y64 = x.double(), X.double(), y.double()
    z = x64 @ X64.T
    ref = (y64 - torch.sigmoid(z)) @ X64 - x64
    ref_lp = (y64 * z - torch.nn.functional.softplus(z, threshold=1e9)).sum(1) - 0.5 * (x64 * x64).sum(1)
    # the tensor-core path's tolerances: 1e-4 of a chain's largest gradient element
    # and of the largest log p
    err = (g - ref).abs().amax(1) / ref.abs().amax(1)
    assert (err[acc] < 1e-4).all()
    assert ((lp - ref_lp).abs()[acc] < 1e-4 * ref_lp.abs().max()).all()
