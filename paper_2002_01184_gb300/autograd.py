"""torch.autograd binding of the batched target log-density.

``TargetLogProb.apply(x, target)`` returns log p(x_c) for every chain row of
x [C, D].  The forward call returns the gradient with it, so the gradient
([C, D] floats) is what autograd keeps and the backward call only weights its
rows (``hmc_target_vjp_from_grad``): evaluating the target a second time, as
``hmc_target_vjp`` does, took as long as the forward pass.  Both directions run
in libhmc's kernels.
"""
import torch

from . import hmc


class Target:
    """A target family bound to device tensors (kept alive here)."""

    def __init__(self, kind, dim, P=None, X=None, y=None):
        dev = lambda a: None if a is None else torch.as_tensor(a).cuda().contiguous()
        self.P, self.X, self.y = dev(P), dev(X), dev(y)
        self.dim = int(dim)
        self.c = hmc.make_target(kind, dim, self.P, self.X, self.y)

    def workspace(self, nbytes):
        return torch.empty(max(int(nbytes), 1), dtype=torch.uint8, device="cuda")


class TargetLogProb(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, target):
        x = x.contiguous()
        C = x.shape[0]
        nbytes = hmc.hmc_grad_workspace_bytes(target.c, C)
        ws = target.workspace(nbytes)
        lp = torch.empty(C, dtype=torch.float32, device=x.device)
        g = torch.empty_like(x)
        hmc.hmc_target_log_prob_and_grad(target.c, C, x, lp, g, ws, nbytes)
        # (x too: a backward pass after x was changed in place stays an error)
        ctx.save_for_backward(x, g)
        return lp

    @staticmethod
    def backward(ctx, grad_lp):
        _, g = ctx.saved_tensors
        C, D = g.shape
        dx = torch.empty_like(g)
        w = grad_lp.to(torch.float32).contiguous()
        hmc.hmc_target_vjp_from_grad(C, D, w, g, dx)
        return dx, None


def log_prob(x, target):
    return TargetLogProb.apply(x, target)
