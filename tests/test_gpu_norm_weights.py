"""Norm weights apart from 1, through every kernel that applies them: the row
norms and the embedding or compaction fused with a norm at each row length a lane
holds (bf16 and float32), the projections of a decode step that norm their input
(up to 8, up to 16 sequences; widths whose chunks and bands end unevenly), and
the kernels that take wider rows.

The weights are drawn between 0.5 and 1.5 for each layer and scaled to unit RMS,
so that the logits keep the size that the stated tolerances are for; a weight
taken from a wrong column moves a row by about 0.4 of its size."""

import dataclasses

import pytest
import torch

from paper_2509_01190_gb300 import inputs as I
from tests.helpers import logits_report, need_gpu
from tests.test_gpu_decode import SMALL, SMALL_128, check_generate, run_generate
from tests.test_gpu_decode_rows import NARROW
from tests.test_gpu_forward import SMALL_BF16, SMALL_CLS, check_case, run_case
from tests.test_gpu_masked import check_masked, run_masked
from tests.test_gpu_rows import wide_bound
from tests.test_gpu_varlen import check_varlen, run_varlen_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


@pytest.fixture(autouse=True)
def drawn_norms(monkeypatch):
    plain = I.make_weights

    def make(shape, device="cpu", seed=I.WEIGHT_SEED):
        w = plain(shape, device=device, seed=seed)
        g = torch.Generator().manual_seed(seed + 1)

        def draw(t):
            v = torch.rand(t.numel(), generator=g) + 0.5
            return (v / v.square().mean().sqrt()).to(device=t.device, dtype=t.dtype)

        for lw in w["layers"]:
            lw["attn_norm"], lw["mlp_norm"] = draw(lw["attn_norm"]), draw(lw["mlp_norm"])
        w["final_norm"] = draw(w["final_norm"])
        return w

    monkeypatch.setattr(I, "make_weights", make)


# 64, 65, 128, 129, 256, 257, 512 and 513 vectors a row
@pytest.mark.parametrize("d", [512, 576, 1024, 1088, 2048, 2112, 4096, 4160])
def test_rows_bf16(z, d):
    shape = I.ModelShape("norms-%d" % d, 2, d, 4, 2, 64, 256, 1008)
    check_case(run_case(z, shape, 2, 37, 2.0, seqs=[0, 1]), "bf16", *wide_bound(d))


@pytest.mark.parametrize("d", [256, 272, 512, 528, 1024, 1040, 2048, 2064])
def test_rows_f32(z, d):
    shape = dataclasses.replace(I.TINY_F32, name="norms-f32-%d" % d, d_model=d, n_heads=4, n_kv_heads=2, head_dim=32,
                                ffn_dim=200, vocab=333)
    check_case(run_case(z, shape, 2, 37, 2.0, seqs=[0, 1]), "f32")


def test_classifier_masked_and_packed_rows(z):
    check_case(run_case(z, SMALL_CLS, 3, 50, 2.0, seqs=[0, 2]), "bf16")
    check_masked(run_masked(z, SMALL_BF16, 2, 50, 2.0))
    check_varlen(run_varlen_case(z, SMALL_BF16, [37, 150, 1, 90, 64], 2.0), SMALL_BF16)


@pytest.mark.parametrize("shape,B", [(SMALL, 1), (SMALL, 8), (SMALL, 9), (SMALL, 16), (SMALL, 17), (NARROW, 3),
                                     (SMALL_128, 2)], ids=lambda v: getattr(v, "name", v))
def test_decode(z, shape, B):
    # A projection that norms its input rounds h w to bf16 where the oracle (and a
    # norm kernel) rounds h / rms w.  With weights of 1 the first is exact; with
    # others the two roundings are independent, and their difference adds to the
    # flips that the stated tolerance is for: two roundings of std 2^-9 / sqrt(3)
    # (relative, of random sign) at two norms a layer and the final one, each of
    # which moves a logit by that part of the logits' std 0.02 sqrt(d).
    L, T = 40, 3
    sigma = (2 * (2 * shape.n_layers + 1) / 3) ** 0.5 * 2.0 ** -9 * 0.02 * shape.d_model ** 0.5
    check_generate(z, shape, run_generate(z, shape, B, L, T, 2.0), B, L, T, sigma if B <= 16 else 0.0)


# (the bound of the wide decode steps in test_gpu_decode_rows.py)
@pytest.mark.parametrize("d,B", [(2112, 5), (4160, 2), (8192, 9)])
def test_decode_wide(z, d, B):
    shape = I.ModelShape("wide-bf16", 2, d, 4, 2, 64, 256, 1008)
    r = run_generate(z, shape, B, 20, 3, 1.5)
    for t in range(3):
        ref = r["ores"]["logits"][:, t]
        mx, mean = logits_report(r["step_logits"][:, t], ref)
        floor = 2.0 ** -7 * shape.n_layers ** 0.5 * ref.std()
        assert mean <= floor and mx <= 8 * floor, (t, mx, mean, floor)
