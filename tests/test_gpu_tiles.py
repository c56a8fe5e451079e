"""Kernels at the edges of their tiles, against the CPU checker: weight matrices
that the GEMM tiles (rows cut to the SM count, k split over a cluster) do not
divide evenly, and trees at the edges of the token tiles; prompts at the edges of
the prefill chunks; fp32 rows that do not divide into fours."""

import numpy as np
import pytest
import torch

from cases import build_case
from gpu_util import TOL, check_case, check_compaction, gpu_cache, gpu_model, max_rel_err, run, to_f64

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2608_00814_gb300 import binding as B  # noqa: E402

# hidden, intermediate, q heads, kv heads: the smallest matrices there are; 3, 5 and
# 4 query heads a kv head; gate/up tiles cut so that every SM has one (80 rows); residual
# tiles cut so that every cluster has one (120 rows, the last one shorter)
SHAPES = [(128, 128, 1, 1), (384, 640, 3, 1), (640, 1152, 5, 1), (1152, 384, 8, 2), (128, 11520, 1, 1),
          (4096, 512, 2, 1)]


@pytest.mark.parametrize("hidden,inter,nq,nkv", SHAPES)
def test_gemm_tile_edges(hidden, inter, nq, nkv):
    # weights scaled so that pre-activations stay near unit size at every width
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=nq, n_kv_heads=nkv, n_layers=2, vocab=700,
                init_std=1.0 / hidden ** 0.5, qkv_bias=True)
    model = None
    for T in (1, 16, 17, 65, 128):
        case = build_case("mini-bf16", 3, T=T, plant=0, ctx_len=37, cfg_overrides=over, gain_std=0.1, prefill=False)
        if model is None:
            model, _ = gpu_model(case)
        kv = gpu_cache(case, case.ctx_len + T)
        g = run(model, kv, case.ctx_len, case.tokens, case.parent)
        r = oracle.verify_tree(case.view, case.cache_k64, case.cache_v64, case.ctx_len, case.tokens, case.parent)
        check_case(case, g, r)
        check_compaction(model, kv, case.ctx_len, g)


@pytest.mark.parametrize("kv", ["", "f16"])
@pytest.mark.parametrize("T", [1, 100, 128])
def test_attention_ragged_end_of_long_ranges(T, kv):
    """Three and more key tiles a block, the last one cut by ctx + T: slots past it
    hold NaN and add nothing, and the tiles before it keep their values."""
    ctx = 2500
    over = dict(hidden=256, intermediate=256, n_q_heads=16, n_kv_heads=8, n_layers=2, vocab=700,
                init_std=1.0 / 16, cache_dtype=kv)
    case = build_case("mini-bf16", 7, T=T, plant=0, ctx_len=ctx, cfg_overrides=over, gain_std=0.1, prefill=False)
    model, _ = gpu_model(case)
    cache = gpu_cache(case, ctx + T + 128)
    for l in range(case.cfg.n_layers):
        cache.k[l][ctx:] = float("nan")
        cache.v[l][ctx:] = float("nan")
    r = oracle.verify_tree(case.view, case.cache_k64, case.cache_v64, ctx, case.tokens, case.parent)
    for _ in range(3):
        check_case(case, run(model, cache, ctx, case.tokens, case.parent), r)


@pytest.mark.parametrize("hidden,inter,nq,nkv,d", [
    (66, 130, 4, 2, 18),    # no row of any weight on a 16-byte boundary
    (64, 131, 3, 1, 6),     # down and O a value at a time, QKV and gate/up in fours
    (70, 128, 5, 5, 2),     # the reverse; the smallest head
])
def test_f32_rows_not_in_fours(hidden, inter, nq, nkv, d):
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=nq, n_kv_heads=nkv, head_dim=d, vocab=501)
    for T in (1, 7, 64):
        case = build_case("tiny", 9, T=T, plant=0, ctx_len=T, cfg_overrides=over, gain_std=0.1, prefill=False)
        model, _ = gpu_model(case)
        kv = gpu_cache(case, case.ctx_len + T)
        g = run(model, kv, case.ctx_len, case.tokens, case.parent)
        r = oracle.verify_tree(case.view, case.cache_k64, case.cache_v64, case.ctx_len, case.tokens, case.parent)
        check_case(case, g, r)
        check_compaction(model, kv, case.ctx_len, g)


@pytest.mark.parametrize("hidden,inter,nq,nkv,kv,ctx,n", [
    (256, 512, 4, 2, "", 0, 129),          # the smallest chunk, one token into the second tile
    (256, 512, 4, 2, "", 131, 2049),       # a whole chunk, then one token through the verify kernels
    (256, 512, 4, 2, "f16", 0, 2048 + 130),   # two chunks
    (384, 640, 3, 1, "", 5, 256),          # an odd number of heads
    (640, 1152, 5, 1, "", 0, 385),         # 25 tokens per attention block
])
def test_prefill_chunk_edges(hidden, inter, nq, nkv, kv, ctx, n):
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=nq, n_kv_heads=nkv, n_layers=2, vocab=700,
                init_std=1.0 / hidden ** 0.5, qkv_bias=True, cache_dtype=kv)
    case = build_case("mini-bf16", 5, T=4, plant=0, ctx_len=ctx, cfg_overrides=over, gain_std=0.1, prefill=False)
    model, _ = gpu_model(case)
    prompt = np.random.default_rng(n).integers(0, case.cfg.vocab, size=n)
    cache = gpu_cache(case, ctx + n + 3)
    tok = torch.as_tensor(prompt.astype(np.int32), device="cuda")
    nxt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    B.oos_prefill(model, cache, ctx, tok, n, nxt)
    torch.cuda.synchronize()
    assert B.oos_last_status(model) == B.OOS_OK
    steps, ck, cv = oracle.decode_sequence(case.view, case.cache_k64, case.cache_v64, ctx, prompt.tolist())
    for l in range(case.cfg.n_layers):
        for got, want in ((cache.k[l], ck[l]), (cache.v[l], cv[l])):
            assert max_rel_err(to_f64(case.cfg, got[ctx:ctx + n]), want[ctx:ctx + n]) <= TOL["bf16"], l
            assert not got[ctx + n:].any()     # nothing past the prompt
    if steps[-1]["top1"] - steps[-1]["top2"] > 0.05:
        assert int(nxt.item()) == int(steps[-1]["argmax"])


def test_prefill_reports_a_bad_token_of_any_chunk():
    case = build_case("mini-bf16", 5, T=4, plant=0, ctx_len=0, prefill=False)
    model, _ = gpu_model(case)
    cache = gpu_cache(case, 2400)
    tok = torch.zeros(2400, dtype=torch.int32, device="cuda")
    for at in (7, 2399):
        tok[at] = case.cfg.vocab
        B.oos_prefill(model, cache, 0, tok, 2400, None)
        assert B.oos_last_status(model) == B.OOS_ETREE
        tok[at] = 0
    B.oos_prefill(model, cache, 0, tok, 2400, None)
    assert B.oos_last_status(model) == B.OOS_OK


@pytest.mark.parametrize("hidden,inter,n", [
    (1280, 3072, 2048),   # narrow: few k-blocks a segment
    (2432, 1024, 300),    # a ragged last token tile of every kind
    (2432, 1152, 2048),
    (2432, 4096, 1700),   # many gate/up tiles a pair, the last cut by the prompt
])
def test_prefill_wide_tiles(hidden, inter, n):
    """One layer, seen through q/k/v and the last token; test_gpu_prefill_tiles.py has
    two, and says which tiles it reaches."""
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=16, n_kv_heads=8, n_layers=1, vocab=700,
                init_std=1.0 / hidden ** 0.5)
    case = build_case("mini-bf16", 6, T=4, plant=0, ctx_len=0, cfg_overrides=over, gain_std=0.1, prefill=False)
    model, _ = gpu_model(case)
    prompt = np.random.default_rng(n).integers(0, case.cfg.vocab, size=n).astype(np.int32)
    cache = gpu_cache(case, n)
    nxt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    B.oos_prefill(model, cache, 0, torch.as_tensor(prompt, device="cuda"), n, nxt)
    torch.cuda.synchronize()
    assert B.oos_last_status(model) == B.OOS_OK
    r = oracle.verify_tree(case.view, case.cache_k64, case.cache_v64, 0, prompt, np.arange(n) - 1)
    for got, want in ((cache.k[0], r["tree_k"][0]), (cache.v[0], r["tree_v"][0])):
        assert max_rel_err(to_f64(case.cfg, got), want) <= TOL["bf16"]
    # the layer's own output is seen through the greedy token of the last position
    if r["top1"][-1] - r["top2"][-1] > 0.05:
        assert int(nxt.item()) == int(r["argmax"][-1])


@pytest.mark.parametrize("hidden,inter,nq,nkv,d", [(512, 1536, 8, 4, 64), (514, 1538, 3, 1, 6)])
def test_f32_trees_of_few_nodes(hidden, inter, nq, nkv, d):
    """Every number of tokens that a warp takes at a time, full and in part."""
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=nq, n_kv_heads=nkv, head_dim=d, vocab=501)
    for T in (1, 2, 3, 4, 5, 8, 9):
        case = build_case("tiny", 9, T=T, plant=0, ctx_len=3, cfg_overrides=over, gain_std=0.1, prefill=False)
        model, _ = gpu_model(case)
        kv = gpu_cache(case, case.ctx_len + T)
        g = run(model, kv, case.ctx_len, case.tokens, case.parent)
        r = oracle.verify_tree(case.view, case.cache_k64, case.cache_v64, case.ctx_len, case.tokens, case.parent)
        check_case(case, g, r)
        check_compaction(model, kv, case.ctx_len, g)
