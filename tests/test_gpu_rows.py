"""The row kernels (embedding or compaction with the next RMSNorm, RMSNorm) at
the sizes where they change: residual widths on both sides of each row length a
lane holds (2, 4, 8, 16 vectors), more rows than the resident warps, and packed
batches of more sequences than one (32) and two (1024) rounds of the search for
a row's sequence."""

import dataclasses

import pytest
import torch

from paper_2509_01190_gb300 import inputs as I
from tests.helpers import BF16_MAX_ABS, BF16_MEAN_ABS, need_gpu
from tests.test_gpu_forward import SMALL_BF16, check_case, run_case
from tests.test_gpu_varlen import check_varlen, run_varlen_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


def wide_bound(d):
    """Bound of the bf16 logits of a model of width d, max-abs and mean-abs.  A
    logit is a sum of d products of a unit-RMS row and weights of std 0.02: its
    std is 0.02 sqrt(d), and the bf16 roundings along the path are relative, so
    its error grows alike.  The stated tolerances are those of d 512 (std 0.45,
    0.044 and 0.0044 of it)."""
    std = 0.02 * max(d, 512) ** 0.5
    return BF16_MAX_ABS / 0.4525 * std, BF16_MEAN_ABS / 0.4525 * std


# 152 SMs hold 7296 warps of the kernels for d <= 1024, 4864 up to 2048, 2432
# above: the larger batches have two rows or more for some warps, also after
# the pruning, and a ragged last block.
@pytest.mark.parametrize("d,B,L", [(512, 3, 67), (576, 2, 33), (512, 200, 79), (1024, 190, 81), (1088, 2, 33),
                                   (2048, 161, 63), (2112, 1, 33), (2112, 81, 63), (4096, 2, 35)])
def test_rows_and_norms(z, d, B, L):
    shape = I.ModelShape("rows-%d" % d, 2, d, 4, 2, 64, 256, 1008)
    res = run_case(z, shape, B, L, 2.0, seqs=[0, B - 1])
    check_case(res, "bf16", *wide_bound(d))


@pytest.mark.parametrize("B", [31, 33, 1030])
def test_packed_rows_of_many_sequences(z, B):
    lengths = [1 + (7 * b) % 5 for b in range(B)]
    check_varlen(run_varlen_case(z, SMALL_BF16, lengths, 1.5), SMALL_BF16)


# float rows: 4 elements a vector, so the same lengths at half the width; past
# d 2048 the embedding, the compaction and the norm are kernels of their own.
@pytest.mark.parametrize("d,B,L", [(256, 3, 67), (272, 2, 33), (256, 200, 79), (1024, 161, 63), (1040, 81, 63),
                                   (2048, 2, 33), (2064, 2, 33)])
def test_rows_and_norms_f32(z, d, B, L):
    shape = dataclasses.replace(I.TINY_F32, name="rows-f32-%d" % d, d_model=d, n_heads=4, n_kv_heads=2, head_dim=32,
                                ffn_dim=200, vocab=333)
    check_case(run_case(z, shape, B, L, 2.0, seqs=[0, B - 1]), "f32")


def _off_by_one(t):
    """A copy of t that starts one element past a 16-byte boundary."""
    store = torch.empty(t.numel() + 8, device=t.device, dtype=t.dtype)
    out = store[1:1 + t.numel()].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == t.element_size()
    return out


# The final norm's weights, and a float32 head, may be any view of the caller's: the
# row kernels read them 16 bytes at a time where they can, else one by one (both
# with the weights drawn apart from 1).  The two forms add a row's squares in other
# orders: float32 results agree to its rounding, bf16 ones to the stated tolerance.
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_final_norm_at_any_element(z, dtype):
    shape = SMALL_BF16 if dtype == "bf16" else dataclasses.replace(I.TINY_F32, prune="1")
    B, L = 3, 41
    w = I.make_weights(shape, device="cuda")
    w["final_norm"] = (1 + 0.5 * torch.randn(shape.d_model, device="cuda")).to(w["final_norm"].dtype)
    odd = dict(w, final_norm=_off_by_one(w["final_norm"]))
    if dtype == "f32":
        odd["head"] = _off_by_one(w["head"])
    tok = torch.from_numpy(I.make_tokens(B, L, shape.vocab)).cuda()
    got = {}
    for name, weights in (("aligned", w), ("odd", odd)):
        model = z.Model(z.config_from_shape(shape), weights, B, L)
        sched, _ = z.zsaa_plan(model, L, 1.5)
        rows = [torch.empty(B, sched[-1], shape.vocab, device="cuda")]
        z.zsaa_forward(model, tok, B, L, 1.5, rows[0])
        if dtype == "bf16":
            rows.append(torch.empty(B, sched[-1], shape.vocab, device="cuda"))
            z.zsaa_forward_masked(model, tok, B, L, 1.5, rows[1])
            cache = z.Cache(model, B, L, 1.5, 2)
            for step in range(3):
                rows.append(torch.empty(B, shape.vocab, device="cuda"))
                if step == 0:
                    z.zsaa_prefill(model, cache, tok, rows[-1])
                else:
                    z.zsaa_decode_step(model, cache, tok[:, step].contiguous(), rows[-1])
        z.zsaa_sync(model)
        got[name] = rows
    for a, b in zip(got["aligned"], got["odd"]):
        err = (a - b).abs()
        if dtype == "f32":
            assert err.max() <= 1e-5 * a.abs().max()
        else:
            assert err.max() <= BF16_MAX_ABS and err.mean() <= BF16_MEAN_ABS


# The embedding is read 16 bytes at a time by every kernel that takes token ids.
def test_unaligned_embedding_is_refused(z):
    w = I.make_weights(SMALL_BF16, device="cuda")
    w["embed"] = _off_by_one(w["embed"])
    model = z.Model(z.config_from_shape(SMALL_BF16), w, 1, 20)
    tok = torch.zeros(1, 20, device="cuda", dtype=torch.int32)
    out = torch.empty(1, 20, SMALL_BF16.vocab, device="cuda")
    cache = z.Cache(model, 1, 20, 1.0, 2)
    for call in (lambda: z.zsaa_forward(model, tok, 1, 20, 1.0, out),
                 lambda: z.zsaa_forward_masked(model, tok, 1, 20, 1.0, out),
                 lambda: z.zsaa_forward_varlen(model, tok, [20], 1.0, out),
                 lambda: z.zsaa_prefill(model, cache, tok, out),
                 lambda: z.zsaa_decode_step(model, cache, tok[:, 0].contiguous(), out)):
        with pytest.raises(z.ZsaaError):
            call()
