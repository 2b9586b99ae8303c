"""theta and log psi of a walker do not depend on how many walkers share its
launch: the number of walkers a group of lanes takes (1, 2, 4, 5, 6 or 8, chosen
by B) changes neither a value nor its order of additions, so the first walkers
of every batch come out bit for bit alike.  One B for each choice on 152 SMs,
ragged, hidden widths of every lane shape."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("N,M", [(12, 16), (18, 33), (16, 72), (12, 130), (10, 300)])
def test_walkers_per_group_leave_the_bits(prec, N, M):
    from paper_2103_08804_gb300 import api
    cd = torch.complex128 if prec == 0 else torch.complex64
    params = dev(synth.rbm_params(71 + M, N, M, 0.1), cd)
    spins = dev(synth.sz0_spins(72, 39007, N), torch.int8)
    first, few = None, 61
    for B in (61, 1201, 2003, 4801, 7001, 9001, 12001, 14003, 19001, 39007):
        ctx = api.Context(N, 1, M, B, prec=prec)
        th = torch.empty(B, M, dtype=cd, device="cuda")
        lp = ctx.rbm_logpsi(params, spins[:B], theta_out=th)
        got = host(th)[:few], host(lp)[:few]
        if first is None:
            first = got
        assert all(np.array_equal(a, b) for a, b in zip(got, first))
        W = params[N + M:].reshape(N, M)  # the last walkers, against torch in 64 bits
        s64 = spins[B - few:B].to(torch.complex128)
        ref = s64 @ W.to(torch.complex128) + params[N:N + M].to(torch.complex128)
        assert float((th[B - few:].to(torch.complex128) - ref).abs().max()) < (1e-12 if prec == 0 else 1e-5)
