"""The fused matrix-free CG of mixed contexts at the edges of its tiles and
slices: one walker tile and pairs of them (up to and over 128 walkers in a
CTA, with a ragged last CTA), one and two column passes (2 M under, at and
over 128), one and several 32-site chunks, and slices from one parameter per
CTA (16 threads each) to most of a hundred (4 threads each).  The product
(S + shift I) v against the float64 S v of the same complex64 tanh(theta).
The operands are split to 2^-24 and summed in float32 accumulators that round
by truncation: at most 54 MMAs in a row for 257 walkers, 6e-8 each, 3e-6 of
partial sums that are a few times the largest entry: 2e-5 of it in all."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("Lx,Ly,M", [(4, 1, 1), (6, 1, 64), (34, 1, 63), (8, 8, 65), (10, 10, 129)])
@pytest.mark.parametrize("wpc", [1, 127, 128, 129, 257])
def test_products_at_tile_edges(Lx, Ly, M, wpc):
    from paper_2103_08804_gb300 import api
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    N, B = Lx * Ly, max(n_sm * wpc - 5, 1) if wpc > 1 else 33
    spins = synth.sz0_spins(3 + wpc, B, N)
    t = (synth.rbm_params(5 + M, B, M - 1, 0.4)[:B * M] if M > 1
         else synth.rbm_params(5, B, 1, 0.4)[:B]).reshape(B, M).astype(np.complex64)
    v = synth.rbm_params(9, N, M, 1.0)
    ctx = api.Context(Lx, Ly, M, B, prec=api.MIXED)
    ds, dt, dv = dev(spins, torch.int8), dev(t, torch.complex64), dev(v, torch.complex128)
    got = ctx.sr_sv(ds, dt, dv, shift=0.25)
    ctx.sync_status()
    s, T = dev(spins, torch.float64), dev(t.astype(np.complex128), torch.complex128)
    V = dv[N + M:].reshape(N, M)
    sc = s.to(torch.complex128)
    u = sc @ dv[:N] + T @ dv[N:N + M] + (T * (sc @ V)).sum(1)
    w = u - u.mean()
    cw = T.conj() * w[:, None]
    ref = torch.cat([sc.T @ w, cw.sum(0), (sc.T @ cw).reshape(-1)]) / B + 0.25 * dv
    assert float((got - ref).abs().max() / ref.abs().max()) < 2e-5
