"""log psi is a sum of log cosh over the hidden units, and M log 2 joins it with
the last level of the sum, whose rounding errors are kept."""

from decimal import Decimal

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def logpsi(b, prec, B=45, N=6):
    from paper_2103_08804_gb300 import api
    M = len(b)
    cd = torch.complex128 if prec == 0 else torch.complex64
    p = np.zeros(N + M + N * M, complex)
    p[N:N + M] = b
    spins = np.tile(np.where(np.arange(N) % 2, 1, -1), (B, 1))
    lp = torch.empty(B, dtype=cd, device="cuda")
    ctx = api.Context(N, 1, M, B, prec=prec)
    ctx.rbm_logpsi(dev(p, cd), dev(spins, torch.int8), logpsi_out=lp)
    return host(lp)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("M", [1, 7, 14, 16, 17, 32, 33, 60, 72, 96, 100, 128, 130, 200, 256, 300, 512])
def test_zero_angles_give_m_log_2(M, prec):
    # log cosh 0 = 0 without rounding, so the result is the number nearest to M log 2
    ln2 = Decimal("0.693147180559945309417232121458176568")
    want = float(M * ln2) if prec == 0 else np.float32(float(M * ln2))
    assert np.all(logpsi(np.zeros(M), prec) == want)


@pytest.mark.parametrize("prec", [0, 1])
def test_infinite_sums_stay_infinite(prec):
    b = np.full(32, 0.1)
    b[3] = 1e300 if prec == 0 else 1e38
    b[4:30] = b[3] * (1e8 if prec == 0 else 3)  # the sum passes the largest number
    assert np.all(np.isposinf(logpsi(b, prec).real))
