"""The estimator sums of mixed, matrix-free steps (one tensor-core product,
its border from the pass that writes the operands) at the edges of their
tiles: sites and hidden units under, at and over a 128-block, walkers around
the 8-walker group, the 128-walker chunk and the 512-walker block.  One SR
step with a shift that dominates S makes the update F / shift, so the sums
show in it: F from float64 sums of the same complex64 tanh(theta) and R.  Each
sum carries three bf16 terms (2^-24) and at most 24 truncated additions per
accumulator (6e-8 each), 1.5e-6 of the summed terms, which are of the size of
R; F is c (<O* R>/<R> - <O*>), two such terms: 3e-6 of max |O R| = 1 scale,
and the CG stops at 1e-9."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("Lx,Ly,M", [(4, 1, 1), (8, 8, 127), (16, 8, 128), (13, 10, 129)])
@pytest.mark.parametrize("B", [1, 7, 129, 513, 4000])
def test_sums_at_tile_edges(Lx, Ly, M, B):
    from paper_2103_08804_gb300 import api
    N = Lx * Ly
    P = N + M + N * M
    spins = synth.sz0_spins(3 + B, B, N)
    t = synth.rbm_params(5 + M, B, M, 0.4)[:B * M].reshape(B, M).astype(np.complex64)
    R = (1.0 + 0.3 * synth.rbm_params(7, B, 1, 1.0)[:B]).astype(np.complex64)
    shift, dgamma = 1e6, 0.1
    ctx = api.Context(Lx, Ly, M, 4000, prec=api.MIXED)
    p0 = np.zeros(P, dtype=np.complex64)
    params = dev(p0, torch.complex64)
    ctx.sr_step(params, dev(spins, torch.int8), dev(t, torch.complex64), dev(R, torch.complex64),
                dgamma, shift, cg_tol=1e-9, mode=api.SR_FIT if hasattr(api, "SR_FIT") else 0)
    ctx.sync_status()
    got = host(params).astype(np.complex128) * shift
    s, T = spins.astype(np.float64), t.astype(np.complex128)
    Rd = R.astype(np.complex128)
    O = np.concatenate([s, T, (s[:, :, None] * T[:, None, :]).reshape(B, N * M)], axis=1)
    ob = O.mean(0)
    mR = Rd.mean()
    ratio = min(abs(mR) ** 2 / np.mean(np.abs(Rd) ** 2), 1.0)
    gamma = np.arccos(np.sqrt(ratio))
    c = dgamma * (1.0 if gamma < 1e-8 else gamma / np.tan(gamma))
    F = c * ((O.conj() * Rd[:, None]).mean(0) / mR - ob.conj())
    # the update solves (S + shift) x = F: undo S by one Neumann term
    x = got
    Sx = (O.conj().T @ (O @ x)) / B - ob.conj() * (ob @ x)
    ref = F - Sx / shift
    scale = abs(c) * np.max(np.abs(O))
    assert np.max(np.abs(got - ref)) < 4e-6 * max(scale, abs(c))
