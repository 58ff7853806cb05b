"""The batch autotuner's measurement of the grouped path is of the code that the
grouped launch runs, not of a context's own form of a small logistic regression."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402


# sizes whose data fits one SM's shared memory; both are grouped by the untuned rule
@pytest.mark.parametrize("N,D,C", [(800, 11, 64), (500, 8, 900)])
def test_grouped_time_is_the_grouped_launchs(N, D, C):
    gen = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(N, D, device="cuda", generator=gen)
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    target = H.make_target("logreg", D, X=X, y=y)
    K = 20
    cfg = H.make_config(10, 0.3 / (N * D) ** 0.5, seed=7)
    x = torch.zeros(C, D, device="cuda")
    s = torch.empty(K, C, D, device="cuda")
    batch = H.hmc_batch_create([target], [C], [cfg])
    assert H.hmc_batch_member_path(batch, 0)[0] == 0
    ms = []
    for _ in range(3):
        x.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        H.hmc_batch_sample_chain(batch, [x], [0], [K], [s], [None], [None])
        b.record()
        H.hmc_batch_synchronize(batch)
        ms.append(a.elapsed_time(b) / K)
    H.hmc_batch_destroy(batch)
    tuned = H.hmc_batch_create_autotuned([target], [C], [cfg])
    path, grouped, tensor = H.hmc_batch_member_path(tuned, 0)
    H.hmc_batch_destroy(tuned)
    # the same tiles: within a factor of two (one is 25 times faster than the other
    # where a context runs whole chains)
    assert 0.5 * min(ms) < grouped < 2.0 * min(ms)
    assert path == (1 if tensor < grouped else 0)
