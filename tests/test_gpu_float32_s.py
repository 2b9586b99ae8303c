"""S of float32 contexts: the products conj(t_j) t_j' are rounded to float32 and
their sums keep what a float64 sum would.  Against S in 64 bits from the same
tanh theta, the error is that of the products' roundings alone, which is formed
here (each product with one fused and one plain rounding, summed in float64):
no more than 1.1 of it in the Frobenius norm over 4e5 entries (a compensated
sum that rounds each corrected term once more had left 1.34)."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def expand(s, y, N, M):
    """S from sum_s sigma_i sigma_i' y_jj' (extended indices, (0, 0) left out), without the means."""
    B = len(s)
    se = np.concatenate([np.ones((B, 1)), s], axis=1)
    a = np.einsum("si,sk->sik", se, se).reshape(B, -1)
    g = (a.T @ y.reshape(B, -1)).reshape(N + 1, N + 1, M + 1, M + 1) / B
    full = g.transpose(0, 2, 1, 3).reshape((N + 1) * (M + 1), -1)
    idx = ([i * (M + 1) for i in range(1, N + 1)] + list(range(1, M + 1)) +
           [i * (M + 1) + j for i in range(1, N + 1) for j in range(1, M + 1)])
    return full[np.ix_(idx, idx)]


@pytest.mark.parametrize("N,M,B", [(12, 30, 2048), (20, 29, 3000)])
def test_sums_keep_what_float64_would(N, M, B):
    from paper_2103_08804_gb300 import api
    g = np.random.Generator(np.random.Philox(91))
    spins = synth.sz0_spins(92, B, N)
    t = (0.3 * (g.standard_normal((B, M)) + 1j * g.standard_normal((B, M)))).astype(np.complex64)
    ctx = api.Context(N, 1, M, B, prec=api.FP32, explicit_s=True)
    S = host(ctx.sr_smatrix(dev(spins, torch.int8), dev(t, torch.complex64), 0.0))
    s = spins.astype(float)
    te = np.concatenate([np.ones((B, 1)), t.astype(np.complex128)], axis=1)
    x, y = te.real, te.imag
    exact = te.conj()[:, :, None] * te[:, None, :]

    def r32(v):
        return v.astype(np.float32).astype(np.float64)

    re = r32(x[:, :, None] * x[:, None, :] + r32(y[:, :, None] * y[:, None, :]))
    im = r32(x[:, :, None] * y[:, None, :] - r32(y[:, :, None] * x[:, None, :]))
    want, rounded = expand(s, exact, N, M), expand(s, re + 1j * im, N, M)
    ob = np.concatenate([s, te[:, 1:], (s[:, :, None] * te[:, None, 1:]).reshape(B, -1)], axis=1).mean(0)
    err = np.linalg.norm(S + np.outer(ob.conj(), ob) - want)
    assert err <= 1.1 * np.linalg.norm(rounded - want)
