"""Exchanged amplitudes that leave float32's range carry the phase of the common
factor exactly: sum_m Im theta_m is about 1536 here, whose float32 rounding alone
is 6e-5 rad.  512 hidden units with one site's weights raised by 0.2, sum_m D =
+-205, so that the factor e^{-+205} of that site's antiparallel bonds leaves
float32 and they take the slow product; where it raises the amplitude they are
all of R.  Errors left: 512 factors of three float32 roundings, theta's own
rounding (2^-23 |theta| per unit), both at random: 8 sqrt(512) 2^-23 = 2.2e-5."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from oracle import rbm, target
from oracle.target import State
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def test_slow_product_keeps_the_phase():
    from paper_2103_08804_gb300 import api
    N, M, B, cd = 8, 512, 48, torch.complex64
    g = np.random.Generator(np.random.Philox(101))
    prm = np.zeros(N + M + N * M, dtype=np.complex128)
    prm[N:N + M] = 0.3 + 3.0j + 1e-3 * (g.standard_normal(M) + 1j * g.standard_normal(M))
    W = 1e-4 * (g.standard_normal((N, M)) + 1j * g.standard_normal((N, M)))
    W[2] += 0.2
    prm[N + M:] = W.reshape(-1)
    prm = prm.astype(np.complex64).astype(np.complex128)
    spins = synth.sz0_spins(102, B, N)
    lp = rbm.logpsi(prm, N, M, spins).astype(np.complex64).astype(np.complex128)
    ctx = api.Context(N, 1, M, B, prec=api.FP32)
    one = dev(np.array([1.0 + 0j]), torch.complex128)
    pt, sp = dev(prm, cd), dev(spins, torch.int8)
    R = host(ctx.cheb_local_target(1, ctx.state(pt), None, one, None, -3.0, 2.0, 0.9, sp, dev(lp, cd)))
    ctx.sync_status()
    ref = target.local_target(1, State(prm), None, 1.0, None, N, M, N, 1, 1.0, -3.0, 2.0, 0.9, (0.0, 0.0),
                              spins, lp)
    big = np.abs(ref) > 1e6
    assert big.sum() > 5
    assert np.max(np.abs(R[big] / ref[big] - 1)) < 2.2e-5
