"""Multi-transition launches of the elementwise targets: bit-identical to the
batch's grouped launch (one warp per chain, one tile function per transition)
at the edges of the lane groups, the chains packed into a warp and the CTAs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402

# (kind, dim, chains): dims around 4 x the lane groups and the 128-dim blocks;
# chains around the packing rule, the CTA sizes and one CTA's share
SHAPES = [("std_normal", 1, 1), ("std_normal", 1, 100), ("std_normal", 1, 9730), ("std_normal", 3, 41),
          ("std_normal", 4, 1300), ("std_normal", 5, 2600), ("std_normal", 130, 9), ("std_normal", 520, 17),
          ("funnel", 2, 1217), ("funnel", 8, 63), ("funnel", 9, 5000), ("funnel", 31, 2500), ("funnel", 64, 1300),
          ("funnel", 100, 4096), ("funnel", 101, 5200), ("funnel", 129, 2500), ("funnel", 257, 33),
          ("funnel", 1024, 5)]


def chain(target, cfg, x0, B, K, grouped):
    C, D = x0.shape
    x = x0.clone()
    s = torch.empty(K, C, D, device="cuda")
    e = torch.empty(K, device="cuda")
    a = torch.empty(K, C, dtype=torch.uint8, device="cuda")
    if grouped:
        b = H.hmc_batch_create([target], [C], [cfg])
        H.hmc_batch_sample_chain(b, [x], [B], [K], [s], [e], [a])
        H.hmc_batch_synchronize(b)
        da = H.hmc_read_adaptation(H.hmc_batch_context(b, 0))
        H.hmc_batch_destroy(b)
    else:
        ctx = H.hmc_create(target, C, cfg)
        H.hmc_sample_chain(ctx, x, B, K, s, e, a)
        H.hmc_synchronize(ctx)
        da = H.hmc_read_adaptation(ctx)
        H.hmc_destroy(ctx)
    return x, s, e, a, da


@pytest.mark.parametrize("kind,dim,chains", SHAPES)
@pytest.mark.parametrize("adapt,B,K", [(False, 2, 35), (True, 34, 5)])
def test_chain_launch_equals_grouped_launch(kind, dim, chains, adapt, B, K):
    g = torch.Generator(device="cuda").manual_seed(dim * 10007 + chains)
    x0 = torch.randn(chains, dim, device="cuda", generator=g)
    cfg = H.make_config(4, 0.4 / dim ** 0.25, seed=7, adapt=adapt, target_accept=0.8, num_adapt_steps=B,
                        chain_offset=3)
    target = H.make_target(kind, dim)
    one, ref = chain(target, cfg, x0, B, K, False), chain(target, cfg, x0, B, K, True)
    for u, v in zip(one[:4], ref[:4]):
        assert torch.equal(u, v)
    assert one[4] == ref[4]
    assert 0 < one[3].float().mean().item() <= 1
