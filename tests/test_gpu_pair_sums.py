"""The explicit S of mixed contexts from spin-pair and tanh-pair sums, at the
edges of its tiles: one tile with a handful of columns, pair and column
counts just under, at and over a block (128 Y columns are (M + 1)^2 with
M = 10 and 11; 256 pairs are 1 + N (N + 1) / 2 with N = 22), walker counts
around the 32-walker tile and the 256-walker chunk.  Every entry of S
against the float64 S of the same complex64 tanh(theta): the products
conj(T_j) T_j' are rounded to float32 once (2^-24 relative, as in float32
contexts) and the sums add at most 48 MMAs per float32 accumulator, 1e-8
relative each (5e-7) before the chunks are added with rounding: 2e-6 of the
largest entry in all."""

import numpy as np
import pytest

from gpu_common import dev, host, need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("shape", [(4, 1, 1), (6, 1, 10), (8, 1, 11), (22, 1, 3), (24, 1, 5),
                                   (4, 5, 33), (12, 1, 16)])
@pytest.mark.parametrize("B", [1, 31, 256, 257, 1100])
def test_pair_sums_at_tile_edges(shape, B):
    from paper_2103_08804_gb300 import api
    Lx, Ly, M = shape
    N = Lx * Ly
    spins = synth.sz0_spins(7 + B, B, N)
    t = synth.rbm_params(11 + M, B, M - 1, 0.4)[:B * M].reshape(B, M).astype(np.complex64)
    ctx = api.Context(Lx, Ly, M, 1100, prec=api.MIXED, explicit_s=True)
    S = host(ctx.sr_smatrix(dev(spins, torch.int8), dev(t, torch.complex64), 0.25))
    ctx.sync_status()
    s, T = spins.astype(np.float64), t.astype(np.complex128)
    O = np.concatenate([s, T, (s[:, :, None] * T[:, None, :]).reshape(B, N * M)], axis=1)
    ob = O.mean(0)
    ref = O.conj().T @ O / B - np.outer(ob.conj(), ob)
    # the entries before the mean is taken off set the scale of the sums' rounding
    scale = np.max(np.abs(O.conj().T @ O / B))
    assert np.array_equal(S, S.conj().T)
    S[np.diag_indices(len(S))] -= 0.25
    assert np.max(np.abs(S - ref)) < 2e-6 * scale
