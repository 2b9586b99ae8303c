"""Two fits in a row of the 10 x 10 lattice with the explicit S in a mixed context
(sweeps, target, S on the tensor cores, factor, refinement): every kernel adds
in a fixed order and the walkers' random stream is counter-based, so a second
run of the same sequence gives the same bits, walkers included, and every
iteration's estimators are finite with the refinement at its tolerance."""

import numpy as np
import pytest

from gpu_common import host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def run():
    from paper_2103_08804_gb300 import api, driver
    L, M, B = 10, 100, 8192
    N = L * L
    E0, a = synth.safe_rescaling(L, L)
    ctx = api.Context(L, L, M, B, prec=api.MIXED, explicit_s=True)
    cfg = driver.SeqConfig(Lx=L, Ly=L, M=M, q=(np.pi, np.pi), n_moments=3, n_iter=12, shift=1e-2, E0=E0, a=a,
                           n_therm=2, n_therm_ref=2, seed=5, solver=api.SOLVE_CHOLESKY, krylov=False)
    seq = driver.Sequence(ctx, cfg, synth.rbm_params(121, N, M, 0.01), synth.sz0_spins(122, B, N),
                          synth.sz0_spins(123, B, N))
    seq.start()
    seq.fit(1)
    seq.fit(2)
    ctx.sync_status()
    out = [host(x) for x in (seq.params, seq.spins, seq.theta, seq.tanh, seq.lp, seq.R, seq.stats, seq.betas)]
    ctx.close()
    return out


def test_a_fit_repeats_bit_for_bit():
    first, again = run(), run()
    assert all(np.array_equal(a, b) for a, b in zip(first, again))
    assert all(np.all(np.isfinite(x)) for x in first)
    stats = first[6][1:]
    assert np.all(stats[:, :, 7] > 0) and np.all(stats[:, :, 6] < 1e-10)
