"""The two-tile tcgen05 attention at the edges of its tiles: 128-query tiles
paired over two heads or over two query blocks of one head, 32-column chunks of
128-key blocks, packed sequences of different lengths."""

import numpy as np
import pytest
import torch

from oracle import zsaa_oracle as O
from paper_2509_01190_gb300 import inputs as I
from tests.helpers import bf16_ulp_close, need_gpu
from tests.test_gpu_forward import SMALL_BF16, SMALL_BF16_128
from tests.test_gpu_ops import _np, _oracle_attention, _qkv
from tests.test_gpu_varlen import check_varlen, run_varlen_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


def _run(z, qkv, B, N, Hq, Hkv, hd, causal, out=None):
    if out is None:
        out = torch.full((B * N, Hq * hd), float("nan"), device="cuda", dtype=torch.bfloat16)
    lse = torch.full((B, Hq, N), float("nan"), device="cuda")
    z.zsaa_op_attention_ex(qkv, B, N, Hq, Hkv, hd, z.ZSAA_BF16, causal, out, lse)
    torch.cuda.synchronize()
    z.zsaa_device_status()
    return out, lse


# Odd ratios pair query blocks (an odd number of blocks leaves a tile empty);
# lengths around the 16-key, 32-column and 128-row edges, many short items.  (Up to
# 64 rows these calls run the mma.sync kernel; see the next test.)
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,N,Hq,Hkv,hd", [(2, 1, 1, 1, 64), (3, 15, 3, 1, 128), (2, 16, 2, 2, 64), (2, 17, 4, 1, 64),
                                           (1, 33, 5, 1, 64), (2, 64, 3, 3, 128), (1, 96, 2, 1, 64), (2, 111, 4, 1, 128),
                                           (1, 127, 1, 1, 128), (2, 129, 3, 1, 64), (1, 255, 2, 2, 128),
                                           (1, 257, 3, 3, 64), (1, 385, 1, 1, 64), (1, 400, 6, 2, 128),
                                           (40, 30, 12, 4, 64), (30, 140, 9, 3, 64)])
def test_attention_tiles(z, B, N, Hq, Hkv, hd, causal):
    qkv = _qkv(B, N, Hq, Hkv, hd, 600 + N, torch.bfloat16)
    out, lse = _run(z, qkv, B, N, Hq, Hkv, hd, causal)
    ref_o, ref_lse, _, _ = _oracle_attention(qkv, B, N, Hq, Hkv, hd, causal=causal)
    got, ref_b = _np(out).reshape(B, N, Hq * hd), O.bf16_round(ref_o)
    # the bounds of test_gpu_ops.py: one bf16 ulp plus 1e-5 of the row's scale
    assert np.all(bf16_ulp_close(got, ref_b, 1, 1e-5 * np.abs(ref_o).max(axis=-1, keepdims=True)))
    assert np.mean(got == ref_b) > 0.95
    np.testing.assert_allclose(_np(lse), ref_lse, rtol=1e-5, atol=1e-4)


# Sequences of up to 64 rows on the tcgen05 kernel, which packed batches with longer
# ones in them give it: alone they reach it in batches past the mma.sync kernel's
# grid (65535 sequences; heads of 128 dims: 512 heads in all).  Lengths around the
# 16-key steps and 32-column chunks of the only key block, next to other sequences'
# rows; a sample of the sequences against the oracle, all of them for being there.
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("N,Hq,Hkv,hd", [(1, 2, 1, 64), (15, 1, 1, 64), (16, 2, 1, 64), (17, 3, 1, 64), (33, 2, 2, 64),
                                         (37, 2, 1, 64), (63, 1, 1, 64), (64, 2, 1, 64), (1, 3, 1, 128),
                                         (17, 2, 1, 128), (37, 3, 1, 128), (48, 4, 1, 128), (64, 1, 1, 128)])
def test_short_sequences_on_tcgen05(z, N, Hq, Hkv, hd, causal):
    B = 65537 if hd == 64 else 513 // Hq + 1
    qkv = torch.randn(B * N, (Hq + 2 * Hkv) * hd, device="cuda", dtype=torch.bfloat16,
                      generator=torch.Generator("cuda").manual_seed(N))
    out, lse = _run(z, qkv, B, N, Hq, Hkv, hd, causal)
    assert torch.isfinite(out).all() and torch.isfinite(lse).all()
    at = torch.tensor(sorted({*range(0, B, max(1, B // 24)), B - 2, B - 1}), device="cuda")
    pick = lambda t: t.view(B, N, -1)[at].reshape(len(at) * N, -1)
    ref_o, ref_lse, _, _ = _oracle_attention(pick(qkv), len(at), N, Hq, Hkv, hd, causal=causal)
    got, ref_b = _np(pick(out)).reshape(ref_o.shape), O.bf16_round(ref_o)
    # the bounds of test_attention_tiles
    assert np.all(bf16_ulp_close(got, ref_b, 1, 1e-5 * np.abs(ref_o).max(axis=-1, keepdims=True)))
    assert np.mean(got == ref_b) > 0.95
    np.testing.assert_allclose(_np(lse[at]), ref_lse, rtol=1e-5, atol=1e-4)


# A packed sequence whose token embeddings are not finite leaves the others as they
# are, bit for bit, in attention, column mass, selection and compaction: packed
# batches of the tcgen05 kernel (one long sequence) and of the mma.sync one (all
# short), first key blocks that end off the 16-key steps.
@pytest.mark.parametrize("lengths", [[37, 21, 300, 13, 150], [37, 21, 40, 13, 64]])
@pytest.mark.parametrize("accel", [1.0, 2.0])
def test_packed_sequences_ignore_each_other(z, lengths, accel):
    for shape in (SMALL_BF16, SMALL_BF16_128):
        w = I.make_weights(shape, device="cuda")
        toks = torch.from_numpy(I.make_tokens(1, sum(lengths), shape.vocab - 2)[0]).cuda()
        bad_rows = [1, 3]
        at = [sum(lengths[:b]) for b in range(len(lengths) + 1)]
        for b in bad_rows:  # NaN and infinity in the last two rows of the embedding
            toks[at[b]:at[b + 1]] = shape.vocab - 2
            toks[at[b] + 1:at[b + 1]:2] = shape.vocab - 1
        model = z.Model(z.config_from_shape(shape), w, len(lengths), max(lengths))
        sched, _ = z.zsaa_plan_varlen(model, lengths, accel)
        n = [s[-1] for s in sched]
        got = []
        for bad in (False, True):
            if bad:
                w["embed"][-2], w["embed"][-1] = float("nan"), float("inf")
                torch.cuda.synchronize()
            logits = torch.empty(sum(n), shape.vocab, device="cuda")
            kept = torch.empty(sum(n), device="cuda", dtype=torch.int32)
            z.zsaa_forward_varlen(model, toks, lengths, accel, logits, kept)
            z.zsaa_sync(model)
            got.append((logits, kept))
        off = 0
        for b, nb in enumerate(n):
            if b not in bad_rows:
                assert torch.equal(got[0][1][off:off + nb], got[1][1][off:off + nb]), b
                assert torch.equal(got[0][0][off:off + nb], got[1][0][off:off + nb]), b
            off += nb
        assert not torch.isfinite(got[1][0]).all()


# Both sides of the lines between this kernel and the mma.sync one of short
# sequences: 64 rows, and for heads of 128 dims 512 heads in all.
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,N,Hq,Hkv,hd", [(3, 63, 4, 2, 64), (3, 64, 4, 2, 64), (3, 65, 4, 2, 64), (64, 48, 32, 8, 64),
                                           (16, 64, 32, 8, 128), (17, 64, 32, 8, 128), (128, 5, 4, 4, 128),
                                           (129, 5, 4, 4, 128)])
def test_attention_of_short_sequences(z, B, N, Hq, Hkv, hd, causal):
    test_attention_tiles(z, B, N, Hq, Hkv, hd, causal)


# Packed lengths of at most 64 rows on average and up to 128 run on the mma.sync
# kernel, longer ones (mean 65, or one of 129) on this.
@pytest.mark.parametrize("lengths", [[128, 1, 60, 30, 64], [64, 64, 64], [64, 64, 67], [129, 1, 20, 30]])
def test_packed_short_sequences(z, lengths):
    for shape in (SMALL_BF16, SMALL_BF16_128):
        check_varlen(run_varlen_case(z, shape, lengths, 1.5), shape)


# An output that allows 16-byte but not 32-byte stores gives the same values.
def test_attention_output_alignment(z):
    B, N, Hq, Hkv, hd = 2, 150, 4, 2, 64
    qkv = _qkv(B, N, Hq, Hkv, hd, 3, torch.bfloat16)
    want, _ = _run(z, qkv, B, N, Hq, Hkv, hd, True)
    store = torch.zeros(B * N * Hq * hd + 16, device="cuda", dtype=torch.bfloat16)
    out = store[8:8 + B * N * Hq * hd].view(B * N, Hq * hd)
    assert out.data_ptr() % 32 == 16
    got, _ = _run(z, qkv, B, N, Hq, Hkv, hd, True, out)
    assert torch.equal(got, want)
    assert not store[:8].any() and not store[8 + B * N * Hq * hd:].any()


# A sequence's last key block reaches into the next sequence's rows: what they
# hold, finite or not, changes nothing.
@pytest.mark.parametrize("N,Hq,Hkv,hd", [(130, 4, 2, 64), (37, 3, 1, 128), (250, 2, 2, 128)])
def test_attention_ignores_the_next_sequence(z, N, Hq, Hkv, hd):
    qkv = _qkv(2, N, Hq, Hkv, hd, 5, torch.bfloat16)
    want, _ = _run(z, qkv, 2, N, Hq, Hkv, hd, True)
    bad = qkv.clone()
    bad[N:] = float("nan")
    bad[N + 1::2] = float("inf")
    got, _ = _run(z, bad, 2, N, Hq, Hkv, hd, True)
    assert torch.equal(got[:N], want[:N])


# Packed lengths through the whole forward: each sequence alone gives the same
# rows, head ratios 1, 3 and 4, lengths of one to four query blocks and of one token.
@pytest.mark.parametrize("heads,kv,hd", [(4, 4, 64), (3, 1, 128), (8, 2, 64)])
def test_varlen_sequences_match_alone(z, heads, kv, hd):
    shape = I.ModelShape("packed", 2, 256, heads, kv, hd, 512, 1008, prune="none")
    w = I.make_weights(shape, device="cuda")
    lengths = [130, 1, 257, 31, 400, 128]
    tok = torch.from_numpy(I.make_tokens(1, sum(lengths), shape.vocab)[0]).cuda()
    model = z.Model(z.config_from_shape(shape), w, len(lengths), max(lengths))
    logits = torch.empty(sum(lengths), shape.vocab, device="cuda")
    z.zsaa_forward_varlen(model, tok, lengths, 1.0, logits)
    z.zsaa_sync(model)
    at = 0
    for n in lengths:
        alone = torch.empty(1, n, shape.vocab, device="cuda")
        z.zsaa_forward(model, tok[at:at + n].contiguous(), 1, n, 1.0, alone)
        z.zsaa_sync(model)
        # other GEMM kernels at other row counts: bf16 storage noise of two layers
        err = (alone[0] - logits[at:at + n]).abs()
        assert err.max() <= 2e-2 and err.mean() <= 2e-3, (n, err.max(), err.mean())
        at += n
