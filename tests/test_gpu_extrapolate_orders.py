"""Linear prediction at the smallest orders, on both sides of the order from
which powers come from tables, and at lengths that fill no table: nothing to
predict, one value, and one block more or less.  A sum of p damped exponentials
is predicted exactly by order p; the fit's condition leaves 1e-8."""

import numpy as np
import pytest

from gpu_common import host, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("p", [1, 2, 3, 7, 8, 9])
@pytest.mark.parametrize("more", [0, 1, 7, 8, 63, 64, 65, 600])
def test_small_orders(p, more):
    from paper_2103_08804_gb300 import api
    N = 6 * p + 10
    z = np.exp(1j * (0.4 + 2 * np.pi * np.arange(p) / p)) * np.linspace(1.0, 0.96, p)
    c = np.linspace(1.0, 0.5, p) * np.exp(0.3j * np.arange(p))
    n = np.arange(N + more)
    mu = (c[:, None] * z[:, None] ** n).sum(0)
    ctx = api.Context(4, 1, 4, 8, prec=api.FP64)
    got = host(ctx.cheb_extrapolate(torch.from_numpy(mu[:N]).cuda(), p, 2 * p, N + more, reg=0.0))
    ctx.sync_status()
    got = got.reshape(-1)
    assert got.shape == mu.shape and np.array_equal(got[:N], mu[:N])
    assert np.max(np.abs(got - mu)) < 1e-8
