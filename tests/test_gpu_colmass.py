"""The tcgen05 column mass at the edges of its tiles: 128-key blocks in pairs,
256-query stages, one or more query heads per tile, against a float64 torch
computation of the same sums."""

import math

import pytest
import torch

from tests.helpers import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


def _reference(x, Hq, Hkv, causal):
    """lse2 [Hq, N] and C [Hkv, N] of one sequence's rows x [N, heads, hd], float64."""
    N, _, hd = x.shape
    lse, C = [], torch.zeros(Hkv, N, device=x.device, dtype=torch.float64)
    for h in range(Hq):
        s = x[:, h] @ x[:, Hq + h // (Hq // Hkv)].T / math.sqrt(hd)
        if causal:
            s = s.masked_fill(torch.ones(N, N, device=x.device).triu(1).bool(), -math.inf)
        l = torch.logsumexp(s, 1)
        C[h // (Hq // Hkv)] += torch.exp(s - l[:, None]).sum(0)
        lse.append(l / math.log(2.0))
    return torch.stack(lse), C


# One key block (N <= 128, the odd last block, few tiles), pairs, a last stage
# of at most 128 queries, halves of the queries (1500 and 1100 rows without the
# mask); (160, 130, ...) has enough tiles for four heads per tile.
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,N,Hq,Hkv,hd", [(3, 1, 4, 2, 64), (2, 33, 3, 1, 128), (5, 128, 4, 1, 64),
                                           (2, 129, 4, 2, 128), (3, 255, 2, 2, 64), (1, 256, 8, 2, 128),
                                           (2, 257, 4, 2, 64), (1, 384, 3, 3, 128), (1, 385, 4, 2, 64),
                                           (1, 640, 4, 1, 128), (1, 1030, 4, 2, 64), (160, 130, 32, 8, 64),
                                           (90, 300, 32, 8, 128),
                                           (1, 1500, 16, 8, 64), (1, 1100, 12, 4, 128)])
def test_colmass_tiles(z, B, N, Hq, Hkv, hd, causal):
    g = torch.Generator(device="cuda").manual_seed(N)
    qkv = torch.randn(B * N, (Hq + 2 * Hkv) * hd, generator=g, device="cuda").to(torch.bfloat16)
    x = qkv.view(B, N, Hq + 2 * Hkv, hd)
    checked = sorted({0, B // 2, B - 1})
    ref = {b: _reference(x[b].double(), Hq, Hkv, causal) for b in checked}
    lse = torch.zeros(B, Hq, N, device="cuda")
    for b in checked:
        lse[b] = ref[b][0].float()
    C = torch.full((B, Hkv, N), float("nan"), device="cuda")
    z.zsaa_op_colmass_ex(qkv, lse, B, N, Hq, Hkv, hd, z.ZSAA_BF16, causal, C)
    again = torch.full_like(C, float("nan"))
    z.zsaa_op_colmass_ex(qkv, lse, B, N, Hq, Hkv, hd, z.ZSAA_BF16, causal, again)
    torch.cuda.synchronize()
    assert torch.equal(C, again)  # a fixed order of sums
    for b in checked:  # the bound of the per-op checks in test_gpu_ops.py
        torch.testing.assert_close(C[b].double(), ref[b][1], rtol=2e-4, atol=1e-5)
