"""tanh theta and log psi next to a zero of cosh theta (theta = i pi / 2 + delta,
|delta| from 1e-2 to 1e-7, all around it, and the other zeros at odd multiples
of i pi / 2): finite, and accurate to the rounding of the given theta.  The
reference is the extended-precision value at the same rounded theta.  tanh: a
denominator of two positive terms, five roundings each plus two units in the
last place of sin, cos and expm1, a division: 16 u.  log psi: the logarithm of
that denominator, 16 u absolute, beside roundings of the sum itself, 4 u |log
psi|."""

import numpy as np
import pytest

from gpu_common import dev, host, logdiff, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def near_nodes(cdtype):
    g = np.random.Generator(np.random.Philox(3))
    z = []
    for k in (-3, -1, 1, 3):
        for r in 10.0 ** -np.arange(2.0, 7.5, 0.5):
            for a in np.concatenate([np.arange(8) * np.pi / 4, g.uniform(0, 2 * np.pi, 8)]):
                z.append(1j * k * np.pi / 2 + r * np.exp(1j * a))
    return np.array(z).astype(cdtype)


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_tanh_and_log_psi_near_a_node(prec):
    from paper_2103_08804_gb300 import api
    cd, u = (torch.complex128, 2.0 ** -53) if prec == 0 else (torch.complex64, 2.0 ** -24)
    th = near_nodes(np.complex128 if prec == 0 else np.complex64)
    N, M = 4, len(th)
    z = th.astype(np.clongdouble)
    ch = np.cosh(z.real) * np.cos(z.imag) + 1j * np.sinh(z.real) * np.sin(z.imag)
    sh = np.sinh(z.real) * np.cos(z.imag) + 1j * np.cosh(z.real) * np.sin(z.imag)
    t_ref = sh / ch
    # one hidden unit of its own per value: a = W = 0, b = theta; walkers of one unit each for log psi
    assert M <= 512 * 2
    for half in np.array_split(np.arange(M), 2):
        m = len(half)
        prm = np.zeros(N + m + N * m, dtype=th.dtype)
        prm[N:N + m] = th[half]
        ctx = api.Context(N, 1, m, 1, prec=prec)
        p, sp = dev(prm, cd), dev(np.array([[1, -1, 1, -1]]), torch.int8)
        theta, T, Ts = (torch.empty(1, m, dtype=cd, device="cuda") for _ in range(3))
        ctx.rbm_logpsi(p, sp, theta_out=theta)
        assert np.array_equal(host(theta)[0], th[half])
        ctx.logderiv(p, sp, theta, tanh_out=T)
        ctx.mc_sweep(p, sp, theta, 0, api.Philox(1, 0), tanh_out=Ts)
        for got in (host(T)[0], host(Ts)[0]):
            assert np.all(np.isfinite(got))
            assert np.max(np.abs(got - t_ref[half]) / np.abs(t_ref[half])) < 16 * u
    lp_ref = np.log(2 * ch)
    ctx = api.Context(N, 1, 1, 1, prec=prec)
    sp = dev(np.array([[1, -1, 1, -1]]), torch.int8)
    for k in range(M):
        prm = np.zeros(N + 1 + N, dtype=th.dtype)
        prm[N] = th[k]
        p = dev(prm, cd)
        theta = torch.empty(1, 1, dtype=cd, device="cuda")
        lp = ctx.rbm_logpsi(p, sp, theta_out=theta)
        lps = torch.empty(1, dtype=cd, device="cuda")
        ctx.mc_sweep(p, sp, theta, 0, api.Philox(1, 0), logpsi_out=lps)
        for got in (host(lp)[0], host(lps)[0]):
            d = logdiff(complex(got), complex(lp_ref[k]))
            assert d < 16 * u + 4 * u * abs(complex(lp_ref[k])), (k, th[k], got, lp_ref[k])


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_walker_at_a_node_moves_on(prec):
    """A walker whose amplitude is all but zero accepts every exchange that
    leads away: its ratio is large, not NaN."""
    from paper_2103_08804_gb300 import api
    N, M, B = 4, 2, 64
    cd = torch.complex128 if prec == 0 else torch.complex64
    prm = np.zeros(N + M + N * M, dtype=np.complex128)
    prm[N:N + M] = [1j * np.pi / 2 - 0.4 + 1e-5, 0.1]
    W = np.zeros((N, M), dtype=np.complex128)
    W[:, 0] = [0.1, -0.1, 0.1, -0.1]  # theta_0 = b_0 + 0.4 on the staggered walker
    prm[N + M:] = W.reshape(-1)
    ctx = api.Context(N, 1, M, B, prec=prec)
    p, sp = dev(prm, cd), dev(np.tile([1, -1, 1, -1], (B, 1)), torch.int8)
    th = torch.empty(B, M, dtype=cd, device="cuda")
    ctx.rbm_logpsi(p, sp, theta_out=th)
    acc = torch.empty(B, dtype=torch.int32, device="cuda")
    T = torch.empty(B, M, dtype=cd, device="cuda")
    lp = torch.empty(B, dtype=cd, device="cuda")
    ctx.mc_sweep(p, sp, th, 2, api.Philox(9, 0), logpsi_out=lp, tanh_out=T, n_accepted=acc)
    assert np.all(host(acc) > 0)
    assert np.all(np.isfinite(host(T))) and np.all(np.isfinite(host(lp)))
