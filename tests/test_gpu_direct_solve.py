"""The direct solve at the edges of its blocks: P one below, at and one above
the 64-row panel, the 256-row tile of the tensor-core update and the 512-row
merged inverse, in every precision (float64 without refinement; float32 on
the FMA pipes; mixed on the tensor cores).  The shifted S is read back with
sr_smatrix and solved in float64 here with the same F (from a first step at
a huge shift, where x = F / shift to 1 / shift): float64 to kappa 2^-53 with
a factor 1e3 for the factorisation's growth; float32 and mixed refine to
|r| <= 1e-12 |F| or stop when the residual no longer halves, so their update
is held to the rounding of the complex64 parameters (2^-24, a factor 4)."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


# (N, M), P = (N + 1)(M + 1) - 1: 59, 64, 65, 254, 257, 510, 512, 1025
SHAPES = [(4, 11), (4, 12), (10, 5), (14, 16), (42, 5), (6, 72), (18, 26), (26, 37)]


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("shape", SHAPES)
def test_direct_solve_at_block_edges(prec, shape):
    from paper_2103_08804_gb300 import api
    N, M = shape
    B, shift = 700, 0.05
    cd = torch.complex128 if prec == 0 else torch.complex64
    g = np.random.Generator(np.random.Philox(N + 100 * M))
    spins = dev(synth.sz0_spins(N, B, N), torch.int8)
    t = dev((0.3 * (g.standard_normal((B, M)) + 1j * g.standard_normal((B, M)))), cd)
    R = dev(1.0 + 0.3 * (g.standard_normal(B) + 1j * g.standard_normal(B)), cd)
    ctx = api.Context(N, 1, M, B, prec=prec, explicit_s=True)
    P = ctx.P
    S = host(ctx.sr_smatrix(spins, t, shift))

    def step(sh):
        p = torch.zeros(P, dtype=cd, device="cuda")
        st = torch.zeros(8, dtype=torch.float64, device="cuda")
        ctx.sr_step(p, spins, t, R, 0.5, sh, solver=api.SOLVE_CHOLESKY, stats_out=st)
        ctx.sync_status()
        return host(p).astype(np.complex128), host(st)

    x, st = step(shift)
    big = 1e9
    F = step(big)[0] * big  # S / big is below 1e-7
    S0 = S - shift * np.eye(P)
    F = F + S0 @ F / big
    ref = np.linalg.solve(S, F)
    kappa = np.linalg.cond(S)
    # F read back through the parameters carries their rounding, which the solve amplifies by
    # at most kappa; the residual norms carry no such factor
    eps = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    r = np.linalg.norm(F - S @ x) / np.linalg.norm(F)
    normS = np.linalg.norm(S, 2) * np.linalg.norm(x) / np.linalg.norm(F)
    assert r < (1e3 * eps if prec == 0 else 4 * eps) * (1 + normS) + 1e-14
    if prec != 0:
        assert st[6] <= 1e-10  # the refinement's own float64 residual
    assert np.linalg.norm(x - ref) <= 1e3 * eps * kappa * np.linalg.norm(ref)
