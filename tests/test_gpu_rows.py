"""The row kernels (embedding or compaction with the next RMSNorm, RMSNorm) at
the sizes where they change: residual widths on both sides of each row length a
lane holds (2, 4, 8, 16 vectors), more rows than the resident warps, and packed
batches of more sequences than one (32) and two (1024) rounds of the search for
a row's sequence."""

import dataclasses

import pytest

from paper_2509_01190_gb300 import inputs as I
from tests.helpers import need_gpu
from tests.test_gpu_forward import SMALL_BF16, check_case, run_case
from tests.test_gpu_varlen import check_varlen, run_varlen_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


# 152 SMs hold 7296 warps of the kernels for d <= 1024, 4864 up to 2048, 2432
# above: the larger batches have two rows or more for some warps, also after
# the pruning, and a ragged last block.
@pytest.mark.parametrize("d,B,L", [(512, 3, 67), (576, 2, 33), (512, 200, 79), (1024, 190, 81), (1088, 2, 33),
                                   (2048, 161, 63), (2112, 1, 33), (2112, 81, 63), (4096, 2, 35)])
def test_rows_and_norms(z, d, B, L):
    shape = I.ModelShape("rows-%d" % d, 2, d, 4, 2, 64, 256, 1008)
    res = run_case(z, shape, B, L, 2.0, seqs=[0, B - 1])
    # A logit is a sum of d products of a unit-RMS row and weights of std 0.02:
    # its std is 0.02 sqrt(d), and the bf16 roundings along the path are relative,
    # so its error grows alike.  The stated tolerance is for widths up to 512
    # (std 0.45): wider models are compared at that scale.
    scale = min(1.0, (512 / d) ** 0.5)
    res["forced_logits"] *= scale
    res["ores"]["logits"] = res["ores"]["logits"] * scale
    check_case(res, "bf16")


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
