"""Spins are int8 at any address: a contiguous view that starts at an odd byte
gives what an aligned copy gives, bit for bit, in every call that reads spins
in words (sites a multiple of 4 and of 16).  Identical inputs take the same
operations in the same order whatever the width of the loads."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("N,M", [(12, 10), (16, 24), (32, 300), (272, 16)])
def test_spins_at_any_byte(prec, N, M):
    from paper_2103_08804_gb300 import api
    B, cd = 131, torch.complex128 if prec == 0 else torch.complex64
    spins0 = synth.sz0_spins(5, B, N)
    params = dev(synth.rbm_params(6, N, M, 0.05), cd)
    g = np.random.Generator(np.random.Philox(7))
    R = dev(1.0 + 0.3 * (g.standard_normal(B) + 1j * g.standard_normal(B)), cd)
    ref = None
    for off in (0, 1, 2, 3, 8):
        buf = torch.zeros(B * N + 64, dtype=torch.int8, device="cuda")
        sp = buf[off:off + B * N].view(B, N)
        sp.copy_(dev(spins0, torch.int8))
        assert sp.data_ptr() % 16 == off
        ctx = api.Context(N, 1, M, B, prec=prec)
        th = torch.empty(B, M, dtype=cd, device="cuda")
        lp = ctx.rbm_logpsi(params, sp, theta_out=th)
        tanh = torch.empty_like(th)
        ctx.mc_sweep(params, sp, th, 1, api.Philox(8, 0), tanh_out=tanh)
        p = params.clone()
        ctx.sr_step(p, sp, tanh, R, 0.5, 1e-2, solver=api.SOLVE_CG, cg_maxit=5, cg_tol=0.0)
        v = torch.ones(ctx.P, dtype=torch.complex128, device="cuda")
        out = ctx.sr_sv(sp, tanh, v, 0.1)
        got = [host(x) for x in (lp, sp, th, p, out)]
        if ref is None:
            ref = got
        assert all(np.array_equal(a, b) for a, b in zip(got, ref))
