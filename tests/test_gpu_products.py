"""The float32 products of the general path at the edges of their tiles (64 and
128 rows, 64 columns, 32-deep steps), for rows that start on 16 bytes and rows
that do not, and the general path's merged elementwise steps."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2002_01184_gb300 import hmc as H  # noqa: E402

U = 2.0 ** -24          # float32 unit round-off


def rand(gen, *shape, offset=0):
    """Normals whose first element lies `offset` floats past an aligned address."""
    n = 1
    for s in shape:
        n *= s
    return torch.randn(n + offset, device="cuda", generator=gen)[offset:].view(*shape)


# 20000 chains: tall tiles; 200: short ones
@pytest.mark.parametrize("C,D", [(1, 1), (63, 3), (64, 32), (65, 33), (129, 64), (200, 65), (127, 130), (300, 511),
                                 (20000, 31), (19999, 68)])
@pytest.mark.parametrize("offset", [0, 1])
def test_gaussian_gradient_at_tile_edges(C, D, offset):
    gen = torch.Generator(device="cuda").manual_seed(C * 1009 + D)
    P = rand(gen, D, D, offset=offset)
    P = (P + P.T).contiguous() if offset == 0 else P          # any square matrix will do
    x = rand(gen, C, D, offset=offset)
    t = H.make_target("corr_gauss", D, P=P)
    lp, g = torch.empty(C, device="cuda"), torch.full((C, D), float("nan"), device="cuda")
    H.hmc_target_log_prob_and_grad(t, C, x, lp, g)
    x64, P64 = x.double(), P.double()
    # a chain of D fused multiply-adds: at most D rounding errors of the partial sums
    bound = (D + 1) * U * (x64.abs() @ P64.abs())
    assert ((g.double() + x64 @ P64).abs() <= bound).all()
    gd = g.double()
    assert ((lp.double() - 0.5 * (x64 * gd).sum(1)).abs() <= (D + 1) * U * (x64 * gd).abs().sum(1)).all()
    w = torch.rand(C, device="cuda", generator=gen)
    nb = H.hmc_target_vjp_workspace_bytes(t, C)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    dx, dx2 = torch.empty_like(g), torch.empty_like(g)
    H.hmc_target_vjp(t, C, x, w, dx, ws, nb)
    H.hmc_target_vjp_from_grad(C, D, w, g, dx2)
    assert torch.equal(dx, w[:, None] * g) and torch.equal(dx2, dx)


@pytest.mark.parametrize("C,N,D", [(1, 1, 1), (63, 65, 5), (65, 64, 33), (129, 511, 64), (200, 1025, 65),
                                   (2500, 700, 30), (70, 9000, 31)])
@pytest.mark.parametrize("offset", [0, 1])
def test_logreg_gradient_at_tile_edges(C, N, D, offset):
    gen = torch.Generator(device="cuda").manual_seed(C * 1009 + N)
    X, x = rand(gen, N, D, offset=offset), rand(gen, C, D, offset=offset) / D ** 0.5
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    t = H.make_target("logreg", D, X=X, y=y)
    nb = H.hmc_grad_workspace_bytes(t, C)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    lp, g = torch.empty(C, device="cuda"), torch.full((C, D), float("nan"), device="cuda")
    H.hmc_target_log_prob_and_grad(t, C, x, lp, g, ws, nb)
    X64, x64, y64 = X.double(), x.double(), y.double()
    z = x64 @ X64.T
    ref = (y64 - torch.sigmoid(z)) @ X64 - x64
    # z is off by at most D roundings of its terms, the residual by a quarter of
    # that and a few roundings, the sum over rows by one rounding per row
    dz = (D + 1) * U * (x64.abs() @ X64.abs().T)
    bound = (0.25 * dz + (N + 8) * U) @ X64.abs() + 4 * U * (x64.abs() + ref.abs())
    assert ((g.double() - ref).abs() <= bound).all()
    terms = y64 * z - torch.nn.functional.softplus(z, threshold=1e9)
    lp_ref = terms.sum(1) - 0.5 * (x64 * x64).sum(1)
    lp_bound = (dz + (N + 8) * U * terms.abs().sum(1, keepdim=True) / N).sum(1) + (D + 2) * U * (x64 * x64).sum(1)
    assert ((lp.double() - lp_ref).abs() <= lp_bound + 4 * U * lp_ref.abs()).all()
    w = torch.rand(C, device="cuda", generator=gen)
    nb = H.hmc_target_vjp_workspace_bytes(t, C)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    dx = torch.empty_like(g)
    H.hmc_target_vjp(t, C, x, w, dx, ws, nb)
    assert torch.equal(dx, w[:, None] * g)


@pytest.mark.parametrize("C,D,L", [(1, 1, 1), (70, 37, 3), (33, 130, 5), (129, 255, 2)])
def test_merged_steps_equal_one_launch_per_operation(C, D, L):
    gen = torch.Generator(device="cuda").manual_seed(D)
    A = torch.randn(D, D, device="cuda", generator=gen)
    P = (A @ A.T / D + 0.1 * torch.eye(D, device="cuda")).contiguous()
    x0 = torch.randn(C, D, device="cuda", generator=gen)
    out = []
    for impl in (H.HMC_IMPL_FUSED, H.HMC_IMPL_PLAIN):
        cfg = H.make_config(L, 0.3 / D ** 0.5, seed=5, adapt=True, num_adapt_steps=4, impl=impl)
        ctx = H.hmc_create(H.make_target("corr_gauss", D, P=P), C, cfg)
        x, s = x0.clone(), torch.empty(5, C, D, device="cuda")
        e, a = torch.empty(5, device="cuda"), torch.empty(5, C, dtype=torch.uint8, device="cuda")
        H.hmc_sample_chain(ctx, x, 3, 5, s, e, a)
        H.hmc_synchronize(ctx)
        H.hmc_destroy(ctx)
        out.append((x, s, e, a))
    for u, v in zip(*out):
        assert torch.equal(u, v)


# one launch per trajectory (clusters of 2 x 2 tiles, a lone chain block, a
# chain or column block past the edge) against one launch per step, which the
# 4300 chains' tiles need: a chain's result does not depend on the others
@pytest.mark.parametrize("D,L", [(260, 1), (260, 5), (320, 4), (512, 3)])
def test_trajectory_launch_equals_step_launches(D, L):
    gen = torch.Generator(device="cuda").manual_seed(D)
    A = torch.randn(D, D, device="cuda", generator=gen, dtype=torch.float64)
    P = (A @ A.T / D + 0.1 * torch.eye(D, device="cuda", dtype=torch.float64)).float().contiguous()
    x0 = torch.randn(4300, D, device="cuda", generator=gen)
    out = []
    for C in (4300, 100, 300, 513):
        cfg = H.make_config(L, 0.05, seed=9)
        ctx = H.hmc_create(H.make_target("corr_gauss", D, P=P), C, cfg)
        x, s = x0[:C].clone(), torch.empty(3, C, D, device="cuda")
        e, a = torch.empty(3, device="cuda"), torch.empty(3, C, dtype=torch.uint8, device="cuda")
        H.hmc_sample_chain(ctx, x, 1, 3, s, e, a)
        H.hmc_synchronize(ctx)
        H.hmc_destroy(ctx)
        out.append((x, s, a))
    assert 0 < out[0][2].float().mean().item()
    for x, s, a in out[1:]:
        C = x.shape[0]
        assert torch.equal(x, out[0][0][:C]) and torch.equal(s, out[0][1][:, :C]) and torch.equal(a, out[0][2][:, :C])


# R X in one to eight tiles of the dims, past one launch's widest tile
@pytest.mark.parametrize("C,N,D", [(40, 5000, 140), (128, 3000, 200), (300, 2500, 301), (90, 2200, 512)])
def test_logreg_tiles_against_float64(C, N, D):
    gen = torch.Generator(device="cuda").manual_seed(D)
    X = torch.randn(N, D, device="cuda", generator=gen)
    y = (torch.rand(N, device="cuda", generator=gen) < 0.5).float()
    x0 = torch.randn(C, D, device="cuda", generator=gen) / D ** 0.5
    cfg = H.make_config(2, 1e-3 / D ** 0.5, seed=3)
    ctx = H.hmc_create(H.make_target("logreg", D, X=X, y=y), C, cfg)
    assert H.hmc_uses_tensor_cores(ctx)
    x = x0.clone()
    H.hmc_bootstrap(ctx, x)
    r = H.hmc_step(ctx, x, 0)
    H.hmc_synchronize(ctx)
    from paper_2002_01184_gb300.sampler import device_view
    g = device_view(r.grad, (C, D), "<f4").clone().double()
    acc = device_view(r.is_accepted, (C,), "|u1").clone().bool()
    H.hmc_destroy(ctx)
    assert acc.any()
    x64 = x.double()
    ref = (y.double() - torch.sigmoid(x64 @ X.double().T)) @ X.double() - x64
    # the tensor-core gradient's tolerance: 1e-4 of each chain's largest element
    err = (g - ref).abs().amax(1) / ref.abs().amax(1)
    assert (err[acc] < 1e-4).all()


# sizes at which tiles of 96 rows fill one wave where 128 leave SMs idle and 64
# need two: the gradient's product, the residuals, the split sum over the rows
@pytest.mark.parametrize("offset", [0, 1])
def test_tiles_of_96_rows(offset):
    for C, D in ((14592, 31), (14591, 68)):
        test_gaussian_gradient_at_tile_edges(C, D, offset)
    for C, N, D in ((2000, 400, 37), (767, 9000, 31)):
        test_logreg_gradient_at_tile_edges(C, N, D, offset)
