"""The Metropolis sweep over many blocks of 64 proposals.  A block can end with
the rows of a proposal in flight that an accepted move has just made parallel
(4% of the blocks of a 10 x 10 lattice); the next block copies into the same
buffer, so a launch over many walkers repeats bit for bit only if that copy has
landed, and a wrong row shows as a wrong decision.

Float64 decisions are those of the oracle (integers exact).  A float32
decision differs where the uniform lies within 1e-5 of the ratio: of 24 walkers
in 400 proposals 0.1, so at most two."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, relerr, torch
from oracle import lattice, rbm, sampler
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("prec,cd,tol", [(0, torch.complex128, 1e-10), (1, torch.complex64, 1e-4)])
@pytest.mark.parametrize("M", [20, 100])
def test_sweep_of_many_blocks(prec, cd, tol, M):
    from paper_2103_08804_gb300 import api
    Lx = Ly = 10
    N, B, n_sweeps, step = 100, 4096, 4, 171
    params = synth.rbm_params(21 + M, N, M, 0.02)
    spins0 = synth.sz0_spins(22, B, N)
    ctx = api.Context(Lx, Ly, M, B, prec=prec)
    pr, first = dev(params, cd), None
    for _ in range(8):
        sp = dev(spins0, torch.int8)
        th = torch.empty(B, M, dtype=cd, device="cuda")
        ctx.rbm_logpsi(pr, sp, theta_out=th)
        acc = torch.empty(B, dtype=torch.int32, device="cuda")
        ctx.mc_sweep(pr, sp, th, n_sweeps, api.Philox(77, 5), n_accepted=acc)
        got = (host(sp), host(acc), host(th))
        if first is None:
            first = got
        assert all(np.array_equal(a, b) for a, b in zip(got, first))
    ids = np.arange(0, B, step)
    s_ref, acc_ref, _ = sampler.mc_sweep(params, N, M, lattice.bonds(Lx, Ly), spins0[ids], n_sweeps, 77, 5,
                                         walker_ids=ids)
    s = first[0][ids]
    same = np.all(s == s_ref, axis=1) & (first[1][ids] == acc_ref)
    assert np.all(same) if prec == 0 else same.sum() >= len(ids) - 2
    assert relerr(first[2], rbm.theta(params, N, M, first[0])) < tol
