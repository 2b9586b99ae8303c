"""The direct solve of the 16 x 16 lattice with 256 hidden units: P = 66,048,
more rows than the y axis of a launch grid holds.  S of 256 walkers is shift I
plus a matrix of rank 255, A^dag A with A = (O - <O>) / sqrt(B), so the
residual of the update is formed in 64 bits without S.  The update comes back
in complex64 parameters (2^-24 |x|) and S is float32-accurate (three bf16
terms and float32 sums: within 2^-22 |S|): residual within 8 x 2^-24 of |F| +
|S| |x|."""

import numpy as np
import pytest

from gpu_common import dev, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def test_more_rows_than_a_grid_axis():
    from paper_2103_08804_gb300 import api
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 150 << 30:
        pytest.skip("S, its factor and the pair sums take 115 GB")
    L, M, B, shift = 16, 256, 256, 0.05
    N = L * L
    g = np.random.Generator(np.random.Philox(41))
    spins = dev(synth.sz0_spins(42, B, N), torch.int8)
    t = dev(0.3 * (g.standard_normal((B, M)) + 1j * g.standard_normal((B, M))), torch.complex64)
    R = dev(1.0 + 0.3 * (g.standard_normal(B) + 1j * g.standard_normal(B)), torch.complex64)
    ctx = api.Context(L, L, M, B, prec=api.MIXED, explicit_s=True)
    p = torch.zeros(ctx.P, dtype=torch.complex64, device="cuda")
    st = torch.zeros(8, dtype=torch.float64, device="cuda")
    ctx.sr_step(p, spins, t, R, 0.5, shift, solver=api.SOLVE_CHOLESKY, stats_out=st)
    ctx.sync_status()
    ctx.close()
    s, t, r = spins.to(torch.complex128), t.to(torch.complex128), R.to(torch.complex128)
    O = torch.cat([s, t, (s[:, :, None] * t[:, None, :]).reshape(B, -1)], dim=1)
    F = st[4] * ((O.conj() * r[:, None]).mean(0) / r.mean() - O.conj().mean(0))
    A = (O - O.mean(0)) / B ** 0.5
    x = p.to(torch.complex128)
    res = F - (A.conj().T @ (A @ x) + shift * x)
    norm_s = torch.linalg.matrix_norm(A @ A.conj().T, 2) + shift
    assert float(res.norm()) <= 8 * 2.0 ** -24 * float(F.norm() + norm_s * x.norm())
    assert float(st[6]) <= 1e-10
