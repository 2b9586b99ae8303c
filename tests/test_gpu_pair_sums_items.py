"""Explicit S of mixed contexts where one CTA of the pair sums takes several tiles
one after another (720 tiles of G on 152 SMs), and where the walkers pass in
several slabs of operands whose sums are added up (45,137 walkers of the 10 x 10
lattice with 100 hidden units: a slab of 44,800 and a ragged one).  Random rows
of S against 64 bits from the same tanh theta, and the same bits again.

A product of three bf16 terms is good to 2^-24, and 48 additions of a chunk
truncate, 2^-24 of the sum of magnitudes each: 3.1e-6 of <|O_k| |O_l|> <= 1."""

import numpy as np
import pytest

from gpu_common import dev, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("N,M,B", [(64, 100, 600), (100, 100, 45137)])
def test_several_items_and_slabs(N, M, B):
    from paper_2103_08804_gb300 import api
    g = torch.Generator(device="cuda")
    g.manual_seed(111)
    t = 0.3 * torch.complex(torch.randn(B, M, device="cuda", generator=g),
                            torch.randn(B, M, device="cuda", generator=g))
    spins = dev(synth.sz0_spins(112, B, N), torch.int8)
    ctx = api.Context(N, 1, M, B, prec=api.MIXED, explicit_s=True)
    S = ctx.sr_smatrix(spins, t, 0.5)
    assert torch.equal(S, ctx.sr_smatrix(spins, t, 0.5))
    ctx.sync_status()
    ctx.close()
    s, T = spins.to(torch.complex128), t.to(torch.complex128)

    def odag(v):  # sum_s v_s O_s
        return torch.cat([s.T @ v, T.T @ v, ((s * v[:, None]).T @ T).reshape(-1)])

    mean = odag(torch.ones(B, dtype=torch.complex128, device="cuda")) / B
    rng = np.random.Generator(np.random.Philox(113))
    rows = [0, N - 1, N, N + M - 1, ctx.P - 1] + list(rng.integers(0, ctx.P, 40))
    for k in map(int, rows):
        if k < N:
            o = s[:, k]
        elif k < N + M:
            o = T[:, k - N]
        else:
            o = s[:, (k - N - M) // M] * T[:, (k - N - M) % M]
        ref = odag(o.conj()) / B - mean[k].conj() * mean
        ref[k] += 0.5
        assert float((S[k] - ref).abs().max()) < 3.1e-6
