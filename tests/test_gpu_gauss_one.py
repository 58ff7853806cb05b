"""The dense Gaussian's one-CTA chains (dim <= 128) against the CTA-pair kernel.
A replica set of two temperatures 1, 1 runs on the pair kernel and exchanges
nothing after odd transitions, so its rows are ordinary chains, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402
from paper_2002_01184_gb300.sampler import device_view  # noqa: E402


# dims around the 32-dim chunks, chains around the 16- and 32-chain shares
@pytest.mark.parametrize("C,D,L", [(2, 4, 1), (34, 32, 3), (62, 36, 2), (66, 100, 5), (130, 128, 16), (1000, 64, 4)])
def test_one_cta_chains_equal_the_pair_kernel(C, D, L):
    gen = torch.Generator(device="cuda").manual_seed(C + D)
    A = torch.randn(D, D, device="cuda", generator=gen, dtype=torch.float64)
    P = (A @ A.T / D + 0.1 * torch.eye(D, device="cuda", dtype=torch.float64)).float().contiguous()
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    target = H.make_target("corr_gauss", D, P=P)
    cfg = H.make_config(L, 0.4 / D ** 0.25, seed=17)
    one, pair = H.hmc_create(target, C, cfg), H.hmc_remc_create(target, C // 2, [1.0, 1.0], cfg)
    out = []
    for ctx in (one, pair):
        x = x0.clone()
        H.hmc_bootstrap(ctx, x)
        got = []
        for t in (1, 3, 5, 7):
            r = H.hmc_step(ctx, x, t)
            H.hmc_synchronize(ctx)
            got += [x.clone()] + [device_view(p, s, f).clone() for p, s, f in (
                (r.target_log_prob, (C,), "<f4"), (r.grad, (C, D), "<f4"), (r.is_accepted, (C,), "|u1"),
                (r.log_accept_ratio, (C,), "<f4"))]
        out.append(got)
        H.hmc_destroy(ctx)
    for u, v in zip(*out):
        assert torch.equal(u, v)
    # whole chains in one launch equal the steps
    ctx = H.hmc_create(target, C, cfg)
    x, s = x0.clone(), torch.empty(8, C, D, device="cuda")
    H.hmc_sample_chain(ctx, x, 0, 8, s)
    H.hmc_synchronize(ctx)
    H.hmc_bootstrap(ctx, x0)
    y = x0.clone()
    for t in range(8):
        H.hmc_step(ctx, y, t)
        assert torch.equal(y, s[t])
    H.hmc_destroy(ctx)
    assert torch.equal(x, y)
