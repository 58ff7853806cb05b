"""Multi-transition launches of the elementwise targets and of small logistic
regressions: bit-identical to the batch's grouped launch (one tile function per
transition) at the edges of the lane groups, the chains packed into a warp, the
row blocks and the CTAs."""
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
    check_equal(H.make_target(kind, dim), cfg, x0, B, K)


# (rows, dim, chains): rows around 16-row blocks and 256-row passes, dims around
# the row strides, chains around the groups per CTA; the last does not fit
# shared memory and takes one launch per transition
LOGREG = [(1, 1, 1), (16, 2, 9), (17, 3, 153), (255, 7, 152), (257, 10, 305), (513, 11, 64), (769, 14, 300),
          (800, 11, 70), (1025, 19, 20), (500, 20, 33), (500, 8, 1048), (30, 23, 700), (19, 512, 10), (40, 129, 90),
          (2048, 64, 8)]


@pytest.mark.parametrize("rows,dim,chains", LOGREG)
@pytest.mark.parametrize("adapt,B,K", [(False, 2, 7), (True, 34, 3)])
def test_logreg_chain_launch_equals_grouped_launch(rows, dim, chains, adapt, B, K):
    g = torch.Generator(device="cuda").manual_seed(rows * 10007 + chains)
    X = torch.randn(rows, dim, device="cuda", generator=g)
    y = (torch.rand(rows, device="cuda", generator=g) < 0.5).float()
    x0 = torch.randn(chains, dim, device="cuda", generator=g) / dim ** 0.5
    cfg = H.make_config(3, 0.5 / (rows * dim) ** 0.5, seed=11, adapt=adapt, target_accept=0.8, num_adapt_steps=B,
                        impl=H.HMC_IMPL_FUSED_SIMT)
    check_equal(H.make_target("logreg", dim, X=X, y=y), cfg, x0, B, K)


def check_equal(target, cfg, x0, B, K):
    one, ref = chain(target, cfg, x0, B, K, False), chain(target, cfg, x0, B, K, True)
    for u, v in zip(one[:4], ref[:4]):
        assert torch.equal(u, v)
    assert one[4] == ref[4]
    assert 0 < one[3].float().mean().item() <= 1
