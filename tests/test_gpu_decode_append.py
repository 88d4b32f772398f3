"""A decode step appends each layer's key, value and position at the row of its
step, however early its kernels start (programmatic launch lets them begin
before the previous step has moved the step counter)."""

import pytest
import torch

from paper_2509_01190_gb300 import inputs as I
from tests.helpers import need_gpu
from tests.test_gpu_decode import SMALL, cache_views

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("B,L", [(1, 300), (1, 600), (2, 300)])
def test_appended_positions(z, B, L, graphs):
    T = 12
    model = z.Model(z.config_from_shape(SMALL), I.make_weights(SMALL, device="cuda"), B, L)
    z.zsaa_model_set_graphs(model, graphs)
    cache = z.Cache(model, B, L, 1.0, T)
    tok = torch.from_numpy(I.make_tokens(B, L + T, SMALL.vocab)).cuda()
    prompt = tok[:, :L].contiguous()
    tokens = [tok[:, L + t].clone() for t in range(T)]  # nothing runs between two steps
    lg = torch.empty(B, SMALL.vocab, device="cuda")
    want = torch.arange(L + T, device="cuda", dtype=torch.int32).expand(B, -1)
    wrong = []
    for n in range(3):
        for layer in range(1, SMALL.n_layers + 1):
            cache_views(z, cache, layer, B, SMALL.n_kv_heads, SMALL.head_dim)[3].fill_(-1)
        z.zsaa_prefill(model, cache, prompt, lg)
        for t in range(T):
            z.zsaa_decode_step(model, cache, tokens[t], lg)
        z.zsaa_sync(model)
        for layer in range(1, SMALL.n_layers + 1):
            pos = cache_views(z, cache, layer, B, SMALL.n_kv_heads, SMALL.head_dim)[3]
            if not torch.equal(pos, want):
                wrong.append((n, layer))
            del pos  # a view of the cache's memory
    cache.close()
    model.close()
    assert not wrong, wrong
