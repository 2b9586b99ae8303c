"""The overlap loss as kernels against the same loss as torch operations (the
path a requires_grad target takes) and against float64: walker counts around a
block of 256 and the 128-block grid, every precision, an upstream factor, and
the forms the kernels leave to torch.  The float64 sums keep the loss to the
rounding of its terms: 1e-12 in float64; in float32 the terms carry d to 2^-24
of |log psi| <= 100, 6e-6 each."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, relerr, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 5e-5), (2, 5e-5)])
@pytest.mark.parametrize("B", [1, 255, 257, 33000])
def test_loss_and_gradient_match_tensor_operations(prec, tol, B):
    from paper_2103_08804_gb300 import api, autograd
    N, M = 8, 9
    cd = torch.complex128 if prec == 0 else torch.complex64
    ctx = api.Context(N, 1, M, B, prec=prec)
    spins = dev(synth.sz0_spins(8 + B, B, N), torch.int8)
    p0 = synth.rbm_params(7, N, M, 0.1)
    lp0 = ctx.rbm_logpsi(dev(synth.rbm_params(9, N, M, 0.1), cd), spins)
    R = dev(1.0 + 0.3 * synth.rbm_params(11, B, 1, 1.0)[:B], cd)
    got = []
    for fused in (True, False):
        p = dev(p0, cd).requires_grad_(True)
        r = R.clone().requires_grad_(not fused)
        loss = autograd.overlap_loss(ctx, p, spins, lp0, r)
        (0.5 * loss).backward()
        got.append((loss.detach(), p.grad))
    assert got[0][0].dtype == got[1][0].dtype and got[0][0].shape == got[1][0].shape
    assert got[0][1].dtype == cd
    # the loss is a logarithm of a ratio near one: absolute
    assert abs(float(got[0][0]) - float(got[1][0])) < tol
    scale = max(float(got[1][1].abs().max()), 1e-1)
    assert float((got[0][1] - got[1][1]).abs().max()) < tol * scale


def test_forms_left_to_tensor_operations():
    from paper_2103_08804_gb300 import api, autograd
    N, M, B = 8, 9, 64
    ctx = api.Context(N, 1, M, B, prec=1)
    spins = dev(synth.sz0_spins(8, B, N), torch.int8)
    p = dev(synth.rbm_params(7, N, M, 0.1), torch.complex64)
    lp0 = ctx.rbm_logpsi(dev(synth.rbm_params(9, N, M, 0.1), torch.complex64), spins)
    R = dev(1.0 + 0.3 * synth.rbm_params(11, B, 1, 1.0)[:B], torch.complex64)
    ok = autograd._fused_loss
    assert ok(ctx, p, spins, lp0, R)
    assert not ok(ctx, p, spins, lp0, R.to(torch.complex128))
    assert not ok(ctx, p, spins, lp0, R.real.contiguous())
    assert not ok(ctx, p, spins, lp0, R[:1])
    assert not ok(ctx, p, spins, lp0[::2], R)
    assert not ok(ctx, p, spins, lp0.clone().requires_grad_(True), R)
    want = float(autograd.overlap_loss(ctx, p, spins, lp0, R))
    assert abs(float(autograd.overlap_loss(ctx, p, spins, lp0, R.to(torch.complex128))) - want) < 5e-5
    assert not ok(ctx, p, spins, lp0, R.conj())
