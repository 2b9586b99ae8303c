"""The two forms of the Metropolis sweep (tables through L1; prefetched rows and
replayed lists) are chosen by the tables' size, the hidden units per lane and
the number of walkers, and take the same operations in the same order: a few
walkers run with few others (lists) and with many (L1) end bit for bit alike,
in spins, accepted moves, theta, tanh theta and log psi.  Sizes on either side
of the walker rule for 1, 2 and 4 units a lane, float64 (L1 up to 4 units a
lane, lists from 8) against the oracle."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, relerr, torch
from oracle import lattice, rbm, sampler
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def sweep(Lx, Ly, M, prec, params, spins0, n_sweeps):
    from paper_2103_08804_gb300 import api
    B = len(spins0)
    cd = torch.complex128 if prec == 0 else torch.complex64
    ctx = api.Context(Lx, Ly, M, B, prec=prec)
    sp, pr = dev(spins0, torch.int8), dev(params, cd)
    th, tanh = (torch.empty(B, M, dtype=cd, device="cuda") for _ in range(2))
    ctx.rbm_logpsi(pr, sp, theta_out=th)
    lp = torch.empty(B, dtype=cd, device="cuda")
    acc = torch.empty(B, dtype=torch.int32, device="cuda")
    ctx.mc_sweep(pr, sp, th, n_sweeps, api.Philox(31, 11), logpsi_out=lp, tanh_out=tanh, n_accepted=acc)
    return [host(x) for x in (sp, acc, th, tanh, lp)]


@pytest.mark.parametrize("Lx,Ly,M,many", [(14, 14, 20, 4000), (10, 10, 60, 4000), (8, 8, 128, 10000)])
@pytest.mark.parametrize("n_sweeps", [1, 3])
def test_routes_agree_bit_for_bit(Lx, Ly, M, many, n_sweeps):
    few = 37
    params = synth.rbm_params(51 + M, Lx * Ly, M, 0.02)
    spins = synth.sz0_spins(52, many, Lx * Ly)
    a = sweep(Lx, Ly, M, 1, params, spins[:few], n_sweeps)
    b = sweep(Lx, Ly, M, 1, params, spins, n_sweeps)
    assert all(np.array_equal(x, y[:few]) for x, y in zip(a, b))


@pytest.mark.parametrize("Lx,Ly,M,many", [(90, 1, 128, 1100), (8, 8, 128, 3000), (10, 10, 100, 3000),
                                          (24, 1, 250, 1400)])
def test_routes_where_a_wave_of_l1_is_full(Lx, Ly, M, many):
    test_routes_agree_bit_for_bit(Lx, Ly, M, many, 1)


@pytest.mark.parametrize("Lx,Ly,M", [(12, 1, 30), (6, 6, 60), (6, 4, 100), (8, 1, 200), (6, 1, 300)])
@pytest.mark.parametrize("n_sweeps", [1, 20])
def test_float64_routes(Lx, Ly, M, n_sweeps):
    N, B = Lx * Ly, 21
    params = synth.rbm_params(61 + M, N, M, 0.05)
    spins = synth.sz0_spins(62, B, N)
    s, acc, th, _, _ = sweep(Lx, Ly, M, 0, params, spins, n_sweeps)
    s_ref, acc_ref, _ = sampler.mc_sweep(params, N, M, lattice.bonds(Lx, Ly), spins, n_sweeps, 31, 11,
                                         walker_ids=np.arange(B))
    assert np.array_equal(s, s_ref) and np.array_equal(acc, acc_ref)
    assert relerr(th, rbm.theta(params, N, M, s)) < 1e-10
