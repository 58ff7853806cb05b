"""Forms that the dense Gaussian takes by its dim: the CTA-pair chains past 128
dims (one CTA per 32 chains below) and the persistent NUTS loop past 256 (a
cluster per chain block below)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H, workloads  # noqa: E402
from paper_2002_01184_gb300.sampler import Sampler  # noqa: E402
from tests import test_gpu_nuts_dense as nuts_dense  # noqa: E402


def problem(C, D, L, B, K):
    p = workloads.corr_gauss(dim=D, num_chains=C, num_burnin=B, num_results=K, num_leapfrog=L)
    return p, torch.as_tensor(p.x0).cuda().contiguous()


@pytest.mark.parametrize("cap", [1, 3])
@pytest.mark.parametrize("C,D", [(192, 132), (200, 256)])
def test_pair_launch_cap_splits_the_chain_without_changing_it(C, D, cap):
    L, B, K = 6, 4, 4
    p, x0 = problem(C, D, L, B, K)
    out = []
    for c in (0, cap):
        s = Sampler(p, adapt=True, max_transitions_per_launch=c)
        x = x0.clone()
        got = s.sample_chain(x, B, K)
        assert H.hmc_dominant_kernel_info(s.ctx) == ("k_gauss_pair", C * L * (c or B + K))
        H.hmc_synchronize(s.ctx)
        out.append((x, *got, s.adaptation()))
        s.close()
    assert all(torch.equal(u, v) for u, v in zip(out[0][:4], out[1][:4]))
    assert out[0][4] == out[1][4]


# batches that divide the kept draws, that do not, and one batch per chain
@pytest.mark.parametrize("D,bsize", [(132, 10), (200, 7), (256, 60)])
def test_pair_streaming_equals_stored_trace(D, bsize):
    from oracle import diagnostics as odiag
    p, x0 = problem(300, D, 8, 20, 60)
    s = Sampler(p)
    x = x0.clone()
    samples, eps, _ = s.sample_chain(x, p.num_burnin, p.num_results)
    x2, eps2 = x0.clone(), torch.empty_like(eps)
    mean, m2, ess = torch.empty_like(x2), torch.empty_like(x2), torch.empty(D, device="cuda")
    H.hmc_sample_chain_streaming_ess(s.ctx, x2, p.num_burnin, p.num_results, bsize, mean, m2, ess, eps2)
    H.hmc_synchronize(s.ctx)
    s.close()
    assert torch.equal(x2, x) and torch.equal(eps2, eps)
    smp = samples.double().cpu().numpy()
    ref_mean = smp.mean(axis=0)
    ref_m2 = ((smp - ref_mean) ** 2).sum(axis=0)
    # the tolerances of the streaming tests at smaller dims
    scale = np.abs(smp).max(axis=0) + 1e-6
    assert np.max(np.abs(mean.double().cpu().numpy() - ref_mean) / scale) < 1e-5
    assert np.max(np.abs(m2.double().cpu().numpy() - ref_m2) / (scale ** 2 * p.num_results)) < 1e-5
    np.testing.assert_allclose(ess.double().cpu().numpy(), odiag.batch_means_ess(smp, bsize), rtol=1e-3)


# a ragged second chain tile with one ragged column tile past 256 dims; the widest
@pytest.mark.parametrize("C,D,eps,depth", [(140, 260, 0.25, 5), (40, 512, 0.2, 5)])
def test_wide_nuts_transition_matches_oracle(C, D, eps, depth):
    nuts_dense.test_dense_nuts_transition_matches_oracle(H, "corr_gauss", C, D, 0, eps, depth)


def test_wide_nuts_chain_is_independent_of_the_batch():
    D = 300
    p = nuts_dense.gauss_problem(200, D, 0.2, 6)
    one = nuts_dense.gauss_problem(1, D, 0.2, 6)
    one.x0 = p.x0[150:151].copy()
    out = []
    for q, offset in ((p, 0), (one, 150)):
        s = Sampler(q, adapt=False, proposal=H.HMC_PROPOSAL_NUTS, chain_offset=offset)
        x = torch.as_tensor(q.x0).cuda().contiguous()
        samples, _, _ = s.sample_chain(x, 1, 4)
        H.hmc_synchronize(s.ctx)
        out.append(samples)
        s.close()
    assert torch.equal(out[0][:, 150], out[1][:, 0])
