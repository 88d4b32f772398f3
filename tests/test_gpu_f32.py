"""The float32 kernels at the sizes where their tiling can go wrong: GEMM tiles
of 64 x 64 x 16 with K split over clusters, attention and column-mass tiles of
16, 32 or 64 rows by 64 columns."""

import dataclasses

import numpy as np
import pytest
import torch

from oracle import zsaa_oracle as O
from paper_2509_01190_gb300 import inputs as I
from tests.helpers import accum_bound, need_gpu
from tests.test_gpu_forward import check_case, run_case
from tests.test_gpu_ops import _np, _oracle_attention, _qkv, _rand

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


# K below one stage, off the 16-byte copies (70, 5), split over 2..8 CTAs of a
# cluster (few tiles, deep K) and whole (many tiles); ragged rows and columns.
@pytest.mark.parametrize("M,N,K", [(1, 3, 5), (64, 64, 16), (65, 130, 70), (63, 65, 15), (129, 96, 272),
                                   (20, 200, 1027), (64, 128, 4096), (300, 516, 512), (1500, 1028, 100),
                                   (40, 64, 20), (70, 100, 48)])
@pytest.mark.parametrize("epi", ["store", "resid", "swiglu"])
def test_linear_f32_tiles(z, epi, M, N, K):
    A, W, W2 = (_rand(s, i, dtype=torch.float32) for i, s in enumerate([(M, K), (N, K), (N, K)]))
    H = _rand((M, N), 3, dtype=torch.float32)
    h0 = _np(H)
    e = {"store": z.EPI_STORE, "resid": z.EPI_RESID, "swiglu": z.EPI_SWIGLU}[epi]
    out = H if epi == "resid" else torch.full((M, N), float("nan"), device="cuda")
    z.zsaa_op_linear(A, W, W2 if epi == "swiglu" else None, H if epi == "resid" else None, out, M, N, K,
                     z.ZSAA_F32, e)
    torch.cuda.synchronize()
    acc, u = _np(A) @ _np(W).T, _np(A) @ _np(W2).T
    ref = {"store": acc, "resid": h0 + acc, "swiglu": O.silu(acc) * u}[epi]
    b = accum_bound(_np(A), _np(W))
    tol = {"store": b, "resid": b, "swiglu": 1.1 * np.abs(u) * b
           + np.abs(O.silu(acc)) * accum_bound(_np(A), _np(W2))}[epi]
    # plus the rounding of the epilogue's own few operations
    assert np.all(np.abs(_np(out) - ref) <= tol + 5e-7 * np.abs(ref))


# Every head size of the tiled kernels and one of the row kernels (96), tile
# edges, odd head ratios; the many-head cases take the 64-row tiles.
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,N,Hq,Hkv,hd", [(1, 1, 2, 2, 64), (2, 15, 3, 1, 128), (1, 17, 4, 2, 32), (2, 63, 4, 4, 64),
                                           (1, 65, 2, 1, 128), (1, 130, 6, 2, 32), (4, 193, 24, 8, 64),
                                           (4, 129, 32, 8, 32), (4, 257, 20, 4, 128), (1, 50, 2, 1, 96)])
def test_attention_and_colmass_f32_tiles(z, B, N, Hq, Hkv, hd, causal):
    qkv = _qkv(B, N, Hq, Hkv, hd, 90 + N, torch.float32)
    out = torch.full((B * N, Hq * hd), float("nan"), device="cuda")
    lse = torch.full((B, Hq, N), float("nan"), device="cuda")
    C = torch.full((B, Hkv, N), float("nan"), device="cuda")
    z.zsaa_op_attention_ex(qkv, B, N, Hq, Hkv, hd, z.ZSAA_F32, causal, out, lse)
    z.zsaa_op_colmass_ex(qkv, lse, B, N, Hq, Hkv, hd, z.ZSAA_F32, causal, C)
    torch.cuda.synchronize()
    ref_o, ref_lse, Ps, _ = _oracle_attention(qkv, B, N, Hq, Hkv, hd, causal=causal)
    # the bounds of the float32 checks in test_gpu_ops.py
    np.testing.assert_allclose(_np(out).reshape(B, N, Hq * hd), ref_o, rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(_np(lse), ref_lse, rtol=1e-5, atol=1e-4)
    refC = np.stack([O.column_mass(Ps[b], Hkv) for b in range(B)])
    np.testing.assert_allclose(_np(C), refC, rtol=1e-5, atol=1e-6)


# The QKV projection's fused RoPE for each way a head lies in a 64-column tile
# (hd 16, 64 and 128, odd head counts), and the separate kernel's (hd 48).
@pytest.mark.parametrize("d,heads,kv,hd,L", [(96, 3, 1, 16, 33), (256, 3, 1, 64, 70), (128, 2, 1, 128, 65),
                                             (192, 4, 2, 48, 40), (512, 8, 8, 64, 130)])
def test_forward_f32_head_sizes(z, d, heads, kv, hd, L):
    shape = dataclasses.replace(I.TINY_F32, name="f32-heads", d_model=d, n_heads=heads, n_kv_heads=kv, head_dim=hd,
                                ffn_dim=200, vocab=333)
    check_case(run_case(z, shape, 2, L, 2.0, seqs=[0, 1]), "f32")


# Causal rows do not see later keys, whatever those hold: with a key and value of
# NaN or infinity the rows before are bitwise unchanged (tiles of 64, 32 and 16 rows,
# the poisoned row first, inside and last in its 64-key block).
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("B,N,Hq,Hkv,hd", [(4, 257, 32, 8, 64), (2, 257, 12, 4, 32), (1, 130, 2, 1, 128),
                                           (4, 193, 40, 8, 128), (1, 70, 3, 3, 64), (1, 70, 2, 1, 96)])
def test_attention_f32_hides_later_rows(z, B, N, Hq, Hkv, hd, bad):
    qkv = _qkv(B, N, Hq, Hkv, hd, 17, torch.float32)

    def run(x):
        out = torch.empty(B, N, Hq * hd, device="cuda")
        lse = torch.empty(B, Hq, N, device="cuda")
        z.zsaa_op_attention_ex(x, B, N, Hq, Hkv, hd, z.ZSAA_F32, True, out, lse)
        torch.cuda.synchronize()
        return out, lse

    want, want_lse = run(qkv)
    for j in (5, 31, 64, N - 1):
        x = qkv.clone()
        x.view(B, N, -1)[:, j, Hq * hd:] = bad
        got, lse = run(x)
        assert torch.equal(got[:, :j], want[:, :j]) and torch.equal(lse[:, :, :j], want_lse[:, :, :j]), j
        assert not torch.isfinite(got[:, j]).any()
