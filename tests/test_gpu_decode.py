"""Generation over the pruned KV cache on the GPU (zsaa_cache_create /
zsaa_prefill / zsaa_decode_step) against the oracle's ``generate``.

Small models: the prefill runs with the oracle's kept indices forced (so bf16
near-ties cannot flip a choice), then T teacher-forced decode steps; the
next-token logits of the prefill and of every step must meet the stated bf16
tolerance, the cached keys/values must match the oracle's cache and the
cached positions must be exact.  Full size (1B shape): the oracle's cache is
written into the GPU cache (inputs flow oracle -> GPU only), so one decode
step differs from the oracle only along its own row through the 16 layers,
and its logits must stay within the noise floor used for chained forwards.
"""

import numpy as np
import pytest
import torch

from oracle import zsaa_oracle as O
from paper_2509_01190_gb300 import inputs as I
from tests.helpers import BF16_MAX_ABS, BF16_MEAN_ABS, logits_report, need_gpu, oracle_cfg

pytestmark = pytest.mark.gpu

SMALL = I.ModelShape("small-bf16", 3, 256, 4, 2, 64, 512, 1008)
SMALL_128 = I.ModelShape("small-bf16-hd128", 2, 512, 4, 1, 128, 768, 2000 - 2000 % 16)
SMALL_8 = I.ModelShape("small-bf16-gqa8", 2, 512, 8, 1, 64, 512, 1024)


@pytest.fixture(scope="module")
def z(zlib):
    need_gpu()
    return zlib


class _DevView:
    """A device buffer of the library seen as a torch tensor (no copy)."""

    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"shape": tuple(shape), "typestr": typestr,
                                         "data": (int(ptr), False), "version": 3}


def cache_views(z, cache, layer, B, Hkv, hd):
    info = z.zsaa_cache_layer(cache, layer)
    cap = info["cap"]
    k = torch.as_tensor(_DevView(info["k"], (B, Hkv, cap, hd), "<i2"), device="cuda").view(torch.bfloat16)
    v = torch.as_tensor(_DevView(info["v"], (B, Hkv, cap, hd), "<i2"), device="cuda").view(torch.bfloat16)
    pos = torch.as_tensor(_DevView(info["pos"], (B, cap), "<i4"), device="cuda")
    return info, k, v, pos


def _forced_blocks(prune, sched, idx_by_layer):
    blocks = [np.asarray(idx_by_layer[l], np.int32).reshape(-1) for l in prune if l in idx_by_layer]
    return torch.from_numpy(np.concatenate(blocks)).cuda() if blocks else None


def run_generate(z, shape, B, L, T, accel, seed=42):
    weights = I.make_weights(shape, device="cuda")
    tokens = I.make_tokens(B, L + T, shape.vocab, seed=seed)
    model = z.Model(z.config_from_shape(shape), weights, B, L)
    sched, alpha = z.zsaa_plan(model, L, accel)
    ocfg = oracle_cfg(shape)
    wnp = I.weights_to_numpy(weights)
    ores = O.generate(ocfg, wnp, tokens[:, :L], tokens[:, L:], alpha=alpha)
    pre = ores["prefill"]
    assert pre["schedule"] == sched
    cache = z.Cache(model, B, L, accel, T)
    prune = shape.prune_layers()
    forced = _forced_blocks(prune, sched, pre["idx"])
    tok = torch.from_numpy(tokens.astype(np.int32)).cuda()
    lg0 = torch.empty(B, shape.vocab, device="cuda", dtype=torch.float32)
    z.zsaa_prefill(model, cache, tok[:, :L].contiguous(), lg0, forced_idx=forced)
    steps = []
    for t in range(T):
        lg = torch.empty(B, shape.vocab, device="cuda", dtype=torch.float32)
        z.zsaa_decode_step(model, cache, tok[:, L + t].contiguous(), lg)
        steps.append(lg)
    z.zsaa_sync(model)
    return dict(model=model, cache=cache, sched=sched, ores=ores, tok=tok, forced=forced,
                prefill_logits=lg0.cpu().numpy(), step_logits=np.stack([s.cpu().numpy() for s in steps], 1))


def check_generate(z, shape, res, B, L, T, step_sigma=0.0):
    """step_sigma: std of a further, stated difference of the decode steps' logits."""
    ores = res["ores"]
    mx, mean = logits_report(res["prefill_logits"], ores["prefill"]["logits"][:, -1])
    assert mx <= BF16_MAX_ABS and mean <= BF16_MEAN_ABS, ("prefill", mx, mean)
    for t in range(T):
        mx, mean = logits_report(res["step_logits"][:, t], ores["logits"][:, t])
        assert mx <= BF16_MAX_ABS + 5 * step_sigma and mean <= BF16_MEAN_ABS + 0.8 * step_sigma, ("step", t, mx, mean)
    Hkv, hd = shape.n_kv_heads, shape.head_dim
    for layer in range(1, shape.n_layers + 1):
        info, k, v, pos = cache_views(z, res["cache"], layer, B, Hkv, hd)
        oc = ores["cache"]["layers"][layer]
        n = info["base"] + T
        assert info["base"] == res["sched"][layer - 1] and info["len"] == n
        np.testing.assert_array_equal(pos[:, :n].cpu().numpy(), oc["pos"])
        # oracle cache [B, n, Hkv, hd] -> [B, Hkv, n, hd]
        for got, ref in ((k, oc["k"]), (v, oc["v"])):
            g = got[:, :, :n].float().cpu().numpy().astype(np.float64)
            r = np.transpose(ref, (0, 2, 1, 3))
            err = np.abs(g - r)
            assert err.max() <= 2e-2 * max(1.0, np.abs(r).max()), (layer, err.max())
            # layer 1 sees identical inputs (bf16 flips of the projection
            # only); deeper layers carry the usual 1-ulp rounding drift
            assert err.mean() <= 2.0 ** -7 * np.abs(r).mean(), (layer, err.mean())
            if layer == 1:
                assert np.mean(err == 0) > 0.9, np.mean(err == 0)


@pytest.mark.parametrize("accel", [1.0, 2.0, 4.0])
def test_generate_small(z, accel):
    B, L, T = 3, 61, 5
    res = run_generate(z, SMALL, B, L, T, accel)
    check_generate(z, SMALL, res, B, L, T)
    pruned, full = z.zsaa_cache_bytes(res["cache"])
    assert pruned <= full and (accel == 1.0) == (pruned == full)


@pytest.mark.parametrize("shape", [SMALL_128, SMALL_8], ids=["hd128", "gqa8"])
def test_generate_small_shapes(z, shape):
    B, L, T = 2, 97, 3
    res = run_generate(z, shape, B, L, T, 3.0)
    check_generate(z, shape, res, B, L, T)


def test_decode_graph_replay_matches_eager(z):
    # first pass: step 1 eager, step 2 recorded, later steps replayed; second
    # pass after a new prefill: every step replayed.  Results are bitwise equal.
    B, L, T = 2, 50, 4
    res = run_generate(z, SMALL, B, L, T, 2.0)
    model, cache, tok = res["model"], res["cache"], res["tok"]
    lg0 = torch.empty(B, SMALL.vocab, device="cuda", dtype=torch.float32)
    z.zsaa_prefill(model, cache, tok[:, :L].contiguous(), lg0, forced_idx=res["forced"])
    buf = torch.empty(B, SMALL.vocab, device="cuda", dtype=torch.float32)
    step_tok = torch.empty(B, device="cuda", dtype=torch.int32)
    outs = []
    for t in range(T):
        step_tok.copy_(tok[:, L + t])
        z.zsaa_decode_step(model, cache, step_tok, buf)
        outs.append(buf.cpu().numpy().copy())
    z.zsaa_prefill(model, cache, tok[:, :L].contiguous(), lg0, forced_idx=res["forced"])
    for t in range(T):
        step_tok.copy_(tok[:, L + t])
        z.zsaa_decode_step(model, cache, step_tok, buf)
        np.testing.assert_array_equal(buf.cpu().numpy(), outs[t])
    np.testing.assert_array_equal(np.stack(outs, 1), res["step_logits"])
    z.zsaa_sync(model)


def test_decode_cache_full_and_bad_args(z):
    B, L = 1, 20
    weights = I.make_weights(SMALL, device="cuda")
    model = z.Model(z.config_from_shape(SMALL), weights, B, L)
    cache = z.Cache(model, B, L, 2.0, 2)
    tok = torch.zeros(B, L, device="cuda", dtype=torch.int32)
    lg = torch.empty(B, SMALL.vocab, device="cuda", dtype=torch.float32)
    z.zsaa_prefill(model, cache, tok, lg)
    t1 = torch.zeros(B, device="cuda", dtype=torch.int32)
    z.zsaa_decode_step(model, cache, t1, lg)
    z.zsaa_decode_step(model, cache, t1, lg)
    with pytest.raises(z.ZsaaError):
        z.zsaa_decode_step(model, cache, t1, lg)
    z.zsaa_prefill(model, cache, tok, lg)  # a new prefill empties the generated part
    z.zsaa_decode_step(model, cache, t1, lg)
    z.zsaa_sync(model)
    with pytest.raises(z.ZsaaError):
        z.Cache(model, B + 1, L, 2.0, 2)
    with pytest.raises(z.ZsaaError):
        z.zsaa_cache_layer(cache, SMALL.n_layers + 1)
    cls = I.ModelShape("small-cls", 2, 256, 4, 2, 64, 512, 1008, n_classes=4)
    wc = I.make_weights(cls, device="cuda")
    mc = z.Model(z.config_from_shape(cls), wc, B, L)
    with pytest.raises(z.ZsaaError):
        z.Cache(mc, B, L, 2.0, 2)


def test_generate_full_size_1b_one_step(z):
    wl = I.WORKLOADS["1b"]
    shape = wl["shape"]
    B, L, accel = 2, wl["L"], 4.0
    weights = I.make_weights(shape, device="cuda")
    tokens = I.make_tokens(1, L + 1, shape.vocab)
    model = z.Model(z.config_from_shape(shape), weights, B, L)
    sched, alpha = z.zsaa_plan(model, L, accel)
    wnp = I.weights_to_numpy(weights)
    ores = O.generate(oracle_cfg(shape), wnp, tokens[:, :L], tokens[:, L:], alpha=alpha)
    pre = ores["prefill"]
    cache = z.Cache(model, B, L, accel, 1)
    prune = shape.prune_layers()
    forced = _forced_blocks(prune, sched, {l: np.repeat(pre["idx"][l], B, 0) for l in prune})
    tok = torch.from_numpy(np.repeat(tokens, B, 0).astype(np.int32)).cuda()
    lg = torch.empty(B, shape.vocab, device="cuda", dtype=torch.float32)
    z.zsaa_prefill(model, cache, tok[:, :L].contiguous(), lg, forced_idx=forced)
    z.zsaa_sync(model)
    # the prefill's own cache must be close to the oracle's, positions exact
    for layer in (1, shape.n_layers):
        info, k, v, pos = cache_views(z, cache, layer, B, shape.n_kv_heads, shape.head_dim)
        oc = pre["cache"]["layers"][layer]
        n = info["base"]
        np.testing.assert_array_equal(pos[:, :n].cpu().numpy(), np.repeat(oc["pos"], B, 0))
        r = np.transpose(oc["k"], (0, 2, 1, 3))[0]
        g = k[0, :, :n].float().cpu().numpy()
        # chained through layer-1 bf16 layers: the noise floor of chained forwards
        rel = np.mean(np.abs(g - r)) / np.mean(np.abs(r))
        assert rel <= 2.0 ** -7 * np.sqrt(layer), (layer, rel)
    # teacher forcing: the oracle's cache replaces the GPU's
    for layer in range(1, shape.n_layers + 1):
        info, k, v, pos = cache_views(z, cache, layer, B, shape.n_kv_heads, shape.head_dim)
        oc = pre["cache"]["layers"][layer]
        n = info["base"]
        for dst, src in ((k, oc["k"]), (v, oc["v"])):
            t = torch.from_numpy(np.transpose(src, (0, 2, 1, 3)).astype(np.float32)).to(torch.bfloat16)
            dst[:, :, :n].copy_(t.expand(B, -1, -1, -1).cuda())
    torch.cuda.synchronize()
    step = torch.empty(B, shape.vocab, device="cuda", dtype=torch.float32)
    z.zsaa_decode_step(model, cache, tok[:, L].contiguous(), step)
    z.zsaa_sync(model)
    ref = np.repeat(ores["logits"][:, 0], B, 0)
    got = step.cpu().numpy()
    mx, mean = logits_report(got, ref)
    floor = 2.0 ** -7 * np.sqrt(shape.n_layers) * ref.std()
    assert mean <= floor and mx <= 8 * floor, (mx, mean, floor)
    np.testing.assert_array_equal(got[0], got[1])  # identical sequences, identical rows
