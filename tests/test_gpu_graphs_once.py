"""hmc_graphs_run_once: ordinary launches in graphs that are launched once; the
same chains."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402


@pytest.mark.parametrize("C,N,D", [(150, 2500, 64), (130, 2200, 201), (40, 100, 9)])
@pytest.mark.parametrize("use_graph", [True, False])
def test_chains_are_the_same(C, N, D, use_graph):
    gen = torch.Generator(device="cuda").manual_seed(D)
    X = torch.randn(N, D, device="cuda", generator=gen)
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    x0 = torch.randn(C, D, device="cuda", generator=gen) / D ** 0.5
    cfg = H.make_config(3, 0.3 / (N * D) ** 0.5, seed=3, adapt=True, num_adapt_steps=3, use_graph=use_graph)
    ctx = H.hmc_create(H.make_target("logreg", D, X=X, y=y), C, cfg)
    x, s = x0.clone(), torch.empty(3, C, D, device="cuda")
    out = []
    for once in (None, True, True, False):
        if once is not None:
            H.hmc_graphs_run_once(ctx, once)
        x.copy_(x0)
        H.hmc_sample_chain(ctx, x, 3, 3, s)
        H.hmc_synchronize(ctx)
        out.append((x.clone(), s.clone(), H.hmc_read_adaptation(ctx)))
    with pytest.raises(H.HMCError) as err:
        H.hmc_graphs_run_once(ctx, 2)
    assert err.value.status == H.HMC_E_INVALID
    H.hmc_destroy(ctx)
    for u in out[1:]:
        assert torch.equal(u[0], out[0][0]) and torch.equal(u[1], out[0][1]) and u[2] == out[0][2]
