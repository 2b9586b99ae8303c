"""The walker kernels at the edges of their tiles: theta and log psi over hidden
units from 1 to 512 and sites that are no multiple of anything, the Metropolis
sweep for every number of hidden units per lane, no sweep at all and over 512
proposals (several rounds of accepted-move lists), and the exchange sums of
the local target over the same sizes, small and large theta.

Tolerances as for the parity of these calls elsewhere: float64 1e-10 relative
(integers exact); float32 u = 6e-8, log psi (N + M) u |log psi|, ratios M u, R
1e-4, or 5e-4 where |log psi| is about 66 (45 additions of u |log psi|, for psi
and for the state it is compared with).  A float32 decision differs from the
float64 one where the uniform lies within 1e-5 of the ratio: 0.15 of 24 walkers
in 540 proposals, so at most two of them."""

import numpy as np
import pytest

from gpu_common import dev, host, logdiff, need_gpu, relerr, torch
from oracle import lattice, rbm, sampler, target
from oracle.target import State
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu

PRECS = {"fp64": (0, torch.complex128, 1e-10), "fp32": (1, torch.complex64, 2e-4)}


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N,M", [(4, 1), (6, 33), (10, 127), (12, 512), (18, 257), (100, 100)])
@pytest.mark.parametrize("B", [1, 9, 700])
def test_theta_at_tile_edges(prec, N, M, B):
    from paper_2103_08804_gb300 import api
    p, cd, tol = PRECS[prec]
    params = synth.rbm_params(3 + M, N, M, 0.1)
    spins = synth.sz0_spins(4 + B, B, N)
    ctx = api.Context(N, 1, M, B, prec=p)
    th = torch.empty(B, M, dtype=cd, device="cuda")
    lp = ctx.rbm_logpsi(dev(params, cd), dev(spins, torch.int8), theta_out=th)
    assert relerr(host(th), rbm.theta(params, N, M, spins)) < (1e-12 if p == 0 else 1e-5)
    assert np.max(logdiff(host(lp), rbm.logpsi(params, N, M, spins))) < tol


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("M", [1, 33, 65, 200, 400])
@pytest.mark.parametrize("n_sweeps", [0, 1, 45])
def test_sweep_per_lane_count(prec, M, n_sweeps):
    from paper_2103_08804_gb300 import api
    N, B = 12, 24
    p, cd, tol = PRECS[prec]
    params = synth.rbm_params(7 + M, N, M, 0.1)
    spins0 = synth.sz0_spins(8, B, N)
    ctx = api.Context(N, 1, M, B, prec=p)
    sp, pr = dev(spins0, torch.int8), dev(params, cd)
    th = torch.empty(B, M, dtype=cd, device="cuda")
    ctx.rbm_logpsi(pr, sp, theta_out=th)
    lp = torch.empty(B, dtype=cd, device="cuda")
    tanh = torch.empty(B, M, dtype=cd, device="cuda")
    acc = torch.empty(B, dtype=torch.int32, device="cuda")
    rng = api.Philox(4321, 7)
    ctx.mc_sweep(pr, sp, th, n_sweeps, rng, logpsi_out=lp, tanh_out=tanh, n_accepted=acc)
    s_ref, acc_ref, ctr = sampler.mc_sweep(params, N, M, lattice.bonds(N, 1), spins0, n_sweeps, 4321, 7,
                                           walker_ids=np.arange(B))
    assert ctr == rng.counter
    s = host(sp)
    same = np.all(s == s_ref, axis=1) & (host(acc) == acc_ref)
    assert np.all(same) if p == 0 else same.sum() >= B - 2
    ref_th = rbm.theta(params, N, M, s)
    assert relerr(host(th), ref_th) < (1e-10 if p == 0 else 1e-4)
    assert relerr(host(tanh), np.tanh(ref_th)) < (1e-10 if p == 0 else 1e-4)
    assert np.max(logdiff(host(lp), rbm.logpsi(params, N, M, s))) < tol


@pytest.mark.parametrize("sigma,tol", [(0.1, 1e-4), (1.0, 5e-4)])
@pytest.mark.parametrize("Lx,Ly,M", [(4, 1, 1), (4, 3, 31), (6, 1, 33), (6, 4, 130), (8, 1, 512)])
@pytest.mark.parametrize("n", [1, 2, 3])
def test_exchange_sums_at_tile_edges(Lx, Ly, M, n, sigma, tol):
    from paper_2103_08804_gb300 import api
    N, B, cd = Lx * Ly, 37, torch.complex64
    if sigma == 1.0 and M > 33:
        sigma = 33.0 / M  # the same |log psi|
    q = (np.pi / 2, np.pi) if Ly > 1 else (np.pi / 2, 0.0)
    J, E0, a, Wp = 1.0, -0.75 * len(lattice.bonds(Lx, Ly)), 3.3, 0.9875
    f32 = [synth.rbm_params(k + M, N, M, sigma).astype(np.complex64).astype(np.complex128)
           for k in range(11, 15)]
    psi, psin = f32[0], f32[3]
    prev = State(psi, probe=True) if n == 1 else State(f32[1])
    prev2 = State(psi, probe=True) if n == 2 else State(f32[2])
    spins = synth.sz0_spins(15, B, N)
    bp, bp2 = 0.7 - 0.2j, -0.4 + 0.9j
    ctx = api.Context(Lx, Ly, M, B, prec=1)
    sp = dev(spins, torch.int8)
    lpn = ctx.rbm_logpsi(dev(psin, cd), sp)
    betas = dev(np.array([bp, bp2]), torch.complex128)
    tp, tp2 = dev(prev.params, cd), dev(prev2.params, cd)
    R = ctx.cheb_local_target(n, ctx.state(tp, prev.probe, q), ctx.state(tp2, prev2.probe, q),
                              betas[0:1], betas[1:2], E0, a, Wp, sp, lpn)
    lp_ref = rbm.logpsi(psin, N, M, spins)
    ref = target.local_target(n, prev, prev2, bp, bp2, N, M, Lx, Ly, J, E0, a, Wp, q, spins, lp_ref)
    assert relerr(host(R) * np.exp(host(lpn) - lp_ref), ref) < tol


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("Lx,Ly,M,B", [(10, 10, 130, 41), (28, 28, 40, 5), (32, 32, 33, 3)])
def test_sweep_replays_large_tables_in_slices(prec, Lx, Ly, M, B):
    """Tables over 128 KB: slices of the widest to the narrowest kind, walker
    counts that fill no group, hidden units that end inside a slice."""
    from paper_2103_08804_gb300 import api
    N = Lx * Ly
    p, cd, _ = PRECS[prec]
    params = synth.rbm_params(7 + M, N, M, 0.02)
    spins0 = synth.sz0_spins(8, B, N)
    ctx = api.Context(Lx, Ly, M, B, prec=p)
    sp, pr = dev(spins0, torch.int8), dev(params, cd)
    th = torch.empty(B, M, dtype=cd, device="cuda")
    ctx.rbm_logpsi(pr, sp, theta_out=th)
    rng = api.Philox(4321, 7)
    ctx.mc_sweep(pr, sp, th, 1, rng)
    s_ref, _, _ = sampler.mc_sweep(params, N, M, lattice.bonds(Lx, Ly), spins0, 1, 4321, 7,
                                   walker_ids=np.arange(B))
    s = host(sp)
    same = np.all(s == s_ref, axis=1)
    assert np.all(same) if p == 0 else same.sum() >= B - 2
    assert relerr(host(th), rbm.theta(params, N, M, s)) < (1e-10 if p == 0 else 1e-4)
