"""log psi of the RBM as a differentiable torch operation (Sec. I, Sec. III).

RBMLogPsi.apply(ctx, params, spins) returns log psi(sigma) for each walker
(complex, [B]) from `rbm_logpsi`; its backward is the hand-written VJP
kernel `logpsi_backward`: for a real loss L with upstream gradient
g_s = dL/d conj(log psi_s) (PyTorch's convention for complex tensors), the
parameter gradient is dL/d conj(alpha_k) = sum_s g_s conj(O_k(s)), with
O_k(s) = d log psi_s / d alpha_k (log psi is holomorphic in alpha).

Both directions run in libchebrbm kernels; torch only provides the
autograd bookkeeping.  overlap_loss has kernels of its own for the loss and
its gradient in log psi where its arguments are plain device vectors; as
separate torch operations they cost more host time than the rest of a
gradient takes on the device.
"""

import torch


class RBMLogPsi(torch.autograd.Function):
    @staticmethod
    def forward(fctx, cr_ctx, params, spins):
        B = spins.shape[0]
        theta = torch.empty(B, cr_ctx.M, dtype=cr_ctx.cdtype, device=spins.device)
        lp = cr_ctx.rbm_logpsi(params.detach().contiguous(), spins, theta_out=theta)
        fctx.cr_ctx = cr_ctx
        fctx.save_for_backward(params, spins, theta)
        return lp

    @staticmethod
    def backward(fctx, grad_lp):
        params, spins, theta = fctx.saved_tensors
        c = fctx.cr_ctx
        T = torch.empty_like(theta)
        c.logderiv(params.detach().contiguous(), spins, theta, tanh_out=T)
        g = c.logpsi_backward(params.detach().contiguous(), spins, T,
                              grad_lp.to(c.cdtype).contiguous())
        return None, g, None


def logpsi(cr_ctx, params, spins):
    """Differentiable log psi: complex [B]."""
    return RBMLogPsi.apply(cr_ctx, params, spins)


class RBMOverlapLoss(torch.autograd.Function):
    """overlap_loss with its sums and its gradient in log psi as kernels."""

    @staticmethod
    def forward(fctx, cr_ctx, params, spins, logpsi0, R):
        theta = torch.empty(spins.shape[0], cr_ctx.M, dtype=cr_ctx.cdtype, device=spins.device)
        lp = cr_ctx.rbm_logpsi(params.detach().contiguous(), spins, theta_out=theta)
        loss, sums = cr_ctx.overlap_loss(lp, logpsi0, R)  # lp becomes log psi - log psi_0
        fctx.cr_ctx = cr_ctx
        fctx.save_for_backward(params, spins, theta, lp, R, sums)
        return loss

    @staticmethod
    def backward(fctx, grad_loss):
        params, spins, theta, d, R, sums = fctx.saved_tensors
        c = fctx.cr_ctx
        g_lp = c.overlap_loss_backward(d, R, sums, grad_loss.resolve_neg().contiguous())
        T = torch.empty_like(theta)
        prm = params.detach().contiguous()
        c.logderiv(prm, spins, theta, tanh_out=T)
        return None, c.logpsi_backward(prm, spins, T, g_lp), None, None, None


def _fused_loss(cr_ctx, params, spins, logpsi0, R):
    """Whether the loss can run as kernels: plain contiguous device vectors of
    the context's complex type that no derivative is taken of, outside
    function transforms and tracing.  Everything else (other types, broadcasts,
    gradients or tangents of logpsi0 or R) is left to torch operations."""
    if torch.compiler.is_compiling() or torch.jit.is_tracing() or spins.ndim != 2 or spins.shape[0] == 0:
        return False
    if torch._C._functorch.peek_interpreter_stack() is not None:
        return False
    if torch.autograd.forward_ad._current_level >= 0:
        return False
    return all(type(t) is torch.Tensor and t.dtype == cr_ctx.cdtype and t.device == spins.device
               and t.is_cuda and t.shape == spins.shape[:1] and t.is_contiguous()
               and not t.is_conj() and not t.is_neg() and not t.requires_grad
               for t in (logpsi0, R))


def overlap_loss(cr_ctx, params, spins, logpsi0, R):
    """The self-normalised importance-sampled infidelity of the fit (Sec. III)
    on fixed samples s of |psi_0|^2 (logpsi0 = log psi_0(s), complex):
        L(alpha) = -log( |sum_s w_s R_s|^2 / (sum_s w_s |R_s|^2 sum_s w_s) ),
    w_s = |psi_alpha(s) / psi_0(s)|^2 and R_s = phi_s / psi_alpha(s), given the
    target ratio R0_s = phi_s / psi_0(s) as R.  At alpha = alpha_0 its gradient
    with respect to conj(alpha) is -(<O* R>/<R> - <O*>), the bracket of the
    natural-gradient force F."""
    if _fused_loss(cr_ctx, params, spins, logpsi0, R):
        return RBMOverlapLoss.apply(cr_ctx, params, spins, logpsi0, R)
    lp = logpsi(cr_ctx, params, spins)
    d = lp - logpsi0.to(lp.dtype)                  # log psi_alpha - log psi_0
    w = torch.exp(2.0 * d.real)
    Ra = R * torch.exp(-d)                         # phi / psi_alpha
    num = torch.abs(torch.sum(w * Ra)) ** 2
    den = torch.sum(w * torch.abs(Ra) ** 2) * torch.sum(w)
    return -torch.log(num / den)
