"""The float32 factor of mixed contexts (trailing update on the tensor cores) is
as good as that of float32 contexts (FMA pipes): the residual that one
correction leaves, |F - S x| / |F| after a solve with the factor alone, is the
factor's error times the condition number.  Both factors take the same panels
and subtract in float32, so the two differ by the roundings of the
products only: within a factor 1.5 (they agree to 10% over P = 168 ... 10200;
48 MMAs into one truncating accumulator had left 1.9 on average)."""

import pytest

from gpu_common import need_gpu, torch
from paper_2103_08804_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("N,M", [(20, 40), (36, 60), (64, 64)])
def test_mixed_factor_as_good_as_float32(N, M):
    from paper_2103_08804_gb300 import api
    B = 4096
    spins = torch.from_numpy(synth.sz0_spins(81, B, N)).cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(82)

    def normal(*shape):
        return torch.complex(torch.randn(*shape, device="cuda", generator=g),
                             torch.randn(*shape, device="cuda", generator=g))

    t, R = 0.3 * normal(B, M), 1.0 + 0.3 * normal(B)
    res = []
    for prec in (api.FP32, api.MIXED):
        ctx = api.Context(N, 1, M, B, prec=prec, explicit_s=True)
        p = torch.zeros(ctx.P, dtype=torch.complex64, device="cuda")
        st = torch.zeros(8, dtype=torch.float64, device="cuda")
        ctx.sr_step(p, spins, t, R, 0.5, 1e-3, solver=api.SOLVE_CHOLESKY, cg_maxit=1, stats_out=st)
        ctx.sync_status()
        assert float(st[5]) == 1.0
        res.append(float(st[6]))
        ctx.close()
    assert res[1] < 1.5 * res[0]
