"""The dense Gaussian's one-CTA chains with a single leapfrog step and a fixed
step size: nothing but the step itself lies between one transition's accept
test and the next one's momenta, so the launch of many transitions has to keep
three of them apart.  Bit-identical to one launch per transition."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402


# every SM with a CTA of its own, and a last CTA that is nearly empty; the four
# lane quarters full or nearly so
@pytest.mark.parametrize("C,D", [(4096, 128), (4001, 100), (700, 36)])
def test_single_step_chain_equals_single_transitions(C, D):
    gen = torch.Generator(device="cuda").manual_seed(C + D)
    A = torch.randn(D, D, device="cuda", generator=gen, dtype=torch.float64)
    P = (A @ A.T / D + 0.1 * torch.eye(D, device="cuda", dtype=torch.float64)).float().contiguous()
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    K = 60
    out = []
    for cap in (0, 1):
        cfg = H.make_config(1, 0.9 / D ** 0.25, seed=23, max_transitions_per_launch=cap)
        ctx = H.hmc_create(H.make_target("corr_gauss", D, P=P), C, cfg)
        x, s = x0.clone(), torch.empty(K, C, D, device="cuda")
        a = torch.empty(K, C, dtype=torch.uint8, device="cuda")
        for _ in range(3):
            x.copy_(x0)
            H.hmc_sample_chain(ctx, x, 0, K, s, None, a)
            H.hmc_synchronize(ctx)
            out.append((x.clone(), s.clone(), a.clone()))
        H.hmc_destroy(ctx)
    accepted = out[0][2].float().mean().item()
    assert 0.05 < accepted < 1.0          # decisions of both kinds
    for u in out[1:]:
        for v, w in zip(u, out[0]):
            assert torch.equal(v, w)


# ... and with running moments instead of a trace
@pytest.mark.parametrize("C,D", [(1500, 128), (70, 40)])
def test_single_step_streaming_equals_stored_trace(C, D):
    gen = torch.Generator(device="cuda").manual_seed(C + D)
    A = torch.randn(D, D, device="cuda", generator=gen, dtype=torch.float64)
    P = (A @ A.T / D + 0.1 * torch.eye(D, device="cuda", dtype=torch.float64)).float().contiguous()
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    B, K = 5, 30
    ctx = H.hmc_create(H.make_target("corr_gauss", D, P=P), C, H.make_config(1, 0.9 / D ** 0.25, seed=23))
    x, s = x0.clone(), torch.empty(K, C, D, device="cuda")
    H.hmc_sample_chain(ctx, x, B, K, s)
    y, mean, m2 = x0.clone(), torch.empty_like(x0), torch.empty_like(x0)
    H.hmc_sample_chain_streaming(ctx, y, B, K, mean, m2)
    H.hmc_synchronize(ctx)
    H.hmc_destroy(ctx)
    assert torch.equal(x, y)
    smp = s.double()
    scale = smp.abs().amax(0) + 1e-6
    # the tolerances of the streaming tests
    assert ((mean.double() - smp.mean(0)).abs() / scale).max() < 1e-5
    assert ((m2.double() - (smp - smp.mean(0)).square().sum(0)).abs() / (scale ** 2 * K)).max() < 1e-5
