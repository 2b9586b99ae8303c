"""The iterative refinement of the direct solve stops when a correction brings
the residual below its tolerance; that last correction belongs to the whole
solution, whichever warp of its kernel runs first.  A float64 context keeps the
solution's bits in its parameters (P = 2162, above the size that is solved
without refinement; shift 1e-6, so that each correction is large beside the
rounding): repeated solves give the same bits, and their residual against S
read back is the one the refinement reports, to the rounding of the product
S x (P 2^-53 |S| |x|)."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def test_last_correction_is_whole():
    from paper_2103_08804_gb300 import api
    N, M, B, shift = 20, 102, 700, 1e-6
    g = np.random.Generator(np.random.Philox(31))
    spins = dev(synth.sz0_spins(32, B, N), torch.int8)
    t = dev(0.3 * (g.standard_normal((B, M)) + 1j * g.standard_normal((B, M))), torch.complex128)
    R = dev(1.0 + 0.3 * (g.standard_normal(B) + 1j * g.standard_normal(B)), torch.complex128)
    ctx = api.Context(N, 1, M, B, prec=0, explicit_s=True)
    first = None
    for _ in range(16):
        p = torch.zeros(ctx.P, dtype=torch.complex128, device="cuda")
        st = torch.zeros(8, dtype=torch.float64, device="cuda")
        ctx.sr_step(p, spins, t, R, 0.5, shift, solver=api.SOLVE_CHOLESKY, stats_out=st)
        ctx.sync_status()
        got = (host(p), host(st))
        if first is None:
            first = got
        assert np.array_equal(got[0], first[0]) and np.array_equal(got[1], first[1])
    x, st = first
    # F on the host, from the same samples
    O = np.concatenate([host(spins).astype(float), host(t),
                        (host(spins)[:, :, None] * host(t)[:, None, :]).reshape(B, -1)], axis=1)
    r = host(R)
    F = st[4] * ((O.conj() * r[:, None]).mean(0) / r.mean() - O.conj().mean(0))
    S = host(ctx.sr_smatrix(spins, t, shift))
    normS = np.linalg.norm(S, 2) * np.linalg.norm(x) / np.linalg.norm(F)
    assert np.linalg.norm(F - S @ x) <= (st[6] + ctx.P * 2.0 ** -53 * (1 + normS)) * np.linalg.norm(F)
