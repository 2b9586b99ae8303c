"""The correction step and the extrapolation at the edges of their grids: Gram
matrices of one state, odd and even counts around the 16 that one CTA takes
and up to 512, one corrected moment and more than the recursion's 512 threads;
prediction of order one, one term past the data, and far past it (several
segments of the power tables).  Poles, weights and moments of well-conditioned
pairs as elsewhere: 1e-9 of G_00 (moments 1e-8).  Prediction: roots to 1e-12
taken to the 1500th power, 1e-8 of the largest moment."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from oracle import extrapolate as ex
from oracle import krylov

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.fixture(scope="module")
def ctx():
    from paper_2103_08804_gb300 import api
    return api.Context(4, 1, 4, 8, prec=0)


@pytest.mark.parametrize("Nm,n_out", [(1, 1), (2, 5), (15, 1), (16, 600), (17, 40), (33, 600), (512, 64)])
def test_krylov_at_grid_edges(ctx, Nm, n_out):
    rng = np.random.default_rng(70 + Nm)
    D = 3 * Nm + 1
    X = (rng.standard_normal((D, Nm)) + 1j * rng.standard_normal((D, Nm))) / np.sqrt(2)
    A = rng.standard_normal((D, D)) + 1j * rng.standard_normal((D, D))
    A = (A + A.conj().T) / 2
    e = np.linalg.eigvalsh(A)
    A = (A - e[0] * np.eye(D)) / ((e[-1] - e[0]) / 1.975) - 0.9875 * np.eye(D)
    G = X.conj().T @ X / D
    G = (G + G.conj().T) / 2
    H = X.conj().T @ A @ X / D
    H = (H + H.conj().T) / 2
    mu = torch.zeros(n_out, dtype=torch.complex128, device="cuda")
    poles = torch.zeros(Nm, dtype=torch.float64, device="cuda")
    wts = torch.zeros(Nm, dtype=torch.float64, device="cuda")
    rank = torch.zeros(1, dtype=torch.int32, device="cuda")
    ctx.cheb_krylov(dev(G, torch.complex128), dev(H, torch.complex128), 1e-12, n_out, mu, poles,
                    wts, rank)
    ctx.sync_status()
    assert int(host(rank)[0]) == Nm
    lam, w = krylov.krylov_poles(G, H, cutoff=1e-12)
    order = np.argsort(lam)
    scale = abs(G[0, 0])
    assert np.allclose(host(poles), lam[order], atol=1e-9)
    assert np.allclose(host(wts), w[order], atol=1e-9 * scale)
    assert np.allclose(host(mu), krylov.corrected_moments(G, H, n_out, cutoff=1e-12), atol=1e-8 * scale)


@pytest.mark.parametrize("modes,N,n0,p,n_out", [(1, 6, 2, 1, 7), (1, 6, 2, 1, 700), (5, 60, 20, 10, 61),
                                                (5, 60, 20, 10, 1500)])
def test_extrapolation_at_segment_edges(ctx, modes, N, n0, p, n_out):
    n = np.arange(N)
    th = np.array([0.3, 0.9, 1.7, 2.2, 2.9])[:modes]
    mu = sum((1.0 + k) * 0.999 ** n * np.exp(1j * t * n) for k, t in enumerate(th))
    ref = ex.extrapolate(mu, p, n0, n_out)[0]
    got = host(ctx.cheb_extrapolate(dev(mu[None], torch.complex128), p, n0, n_out))
    got = got.reshape(-1)
    ctx.sync_status()
    assert np.array_equal(got[:N], mu)
    assert np.max(np.abs(got - ref)) < 1e-8 * np.max(np.abs(mu))
