"""Decode steps at the row counts where the step's kernels change: up to 8 and up
to 16 sequences (residual rows normed inside the weight-streaming projections),
17 (norms as kernels of their own); a residual width with fewer 32-wide chunks
than warps; caches of less than one and of several 32-key blocks per warp."""

import pytest

from paper_2509_01190_gb300 import inputs as I
from tests.helpers import BF16_MAX_ABS, BF16_MEAN_ABS, logits_report, need_gpu
from tests.test_gpu_decode import SMALL, SMALL_128, run_generate

pytestmark = pytest.mark.gpu

NARROW = I.ModelShape("narrow-bf16", 2, 128, 2, 2, 64, 192, 1008)


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


@pytest.mark.parametrize("shape,B,L,T,accel", [(SMALL, 1, 7, 3, 1.0), (SMALL, 8, 40, 3, 2.0), (SMALL, 9, 33, 3, 2.0),
                                               (SMALL, 16, 20, 2, 1.5), (SMALL, 17, 20, 2, 1.5),
                                               (NARROW, 3, 31, 4, 1.0), (SMALL, 1, 600, 3, 1.0),
                                               (SMALL_128, 2, 300, 3, 1.0)],
                         ids=lambda v: getattr(v, "name", v))
def test_decode_rows(z, shape, B, L, T, accel):
    r = run_generate(z, shape, B, L, T, accel)
    for t in range(T):
        mx, mean = logits_report(r["step_logits"][:, t], r["ores"]["logits"][:, t])
        assert mx <= BF16_MAX_ABS and mean <= BF16_MEAN_ABS, (t, mx, mean)


# Residual rows of more than 512 16-byte vectors (d 4096): the step embeds and norms
# them in kernels of their own, in front of the folded projections (up to 16
# sequences, d 8192) and of the plain ones.  A logit is a sum of d products of a
# unit-RMS row and weights of std 0.02, so its error grows with its own size: the
# bound is the one of chained forwards, 2^-7 of the logits' std per layer (mean) and
# eight times that (max).
@pytest.mark.parametrize("d,B", [(4160, 2), (5120, 16), (5120, 17), (8192, 3), (8256, 2)])
def test_decode_of_wide_rows(z, d, B):
    shape = I.ModelShape("wide-bf16", 2, d, 4, 2, 64, 256, 1008)
    r = run_generate(z, shape, B, 20, 3, 1.5)
    for got, ref in [(r["prefill_logits"], r["ores"]["prefill"]["logits"][:, -1])] + [
            (r["step_logits"][:, t], r["ores"]["logits"][:, t]) for t in range(3)]:
        mx, mean = logits_report(got, ref)
        floor = 2.0 ** -7 * shape.n_layers ** 0.5 * ref.std()
        assert mean <= floor and mx <= 8 * floor, (mx, mean, floor)
