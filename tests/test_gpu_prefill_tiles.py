"""Both kinds of prefill tiles, element by element: a second layer, whose K and V show
every row of the first one's attention, O, gate/up and down.  Each case asks which tiles
its GEMMs take, so that another choice cannot empty it."""

import ctypes

import numpy as np
import pytest
import torch

from cases import build_case
from gpu_util import TOL, gpu_cache, gpu_model, max_rel_err, to_f64

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2608_00814_gb300 import binding as B  # noqa: E402

GEMMS = dict(qkv=B.OOS_STAGE_QKV, o=B.OOS_STAGE_O, gu=B.OOS_STAGE_GATE_UP, down=B.OOS_STAGE_DOWN)


def tiles(model, gemm, n):
    f = B.lib().oos_prefill_tiles
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32, ctypes.c_int32], ctypes.c_int32
    return f(model.handle, 0, GEMMS[gemm], n)


@pytest.mark.parametrize("hidden,inter,nq,nkv,kv,bias,n,pairs,verify", [
    # 25 heads: the last tile's second half past the matrices; bias; binary16 K and V
    (2432, 3072, 15, 5, "f16", True, 1280, ["qkv", "gu"], ["o"]),
    (2432, 3072, 15, 5, "", False, 1153, ["qkv"], ["o", "gu"]),     # one token in the last token tile
    (2432, 8192, 4, 2, "", False, 1792, ["gu", "down"], ["o"]),     # one tile a pair; gate/up six
    (4096, 4096, 2, 1, "", True, 2048, ["gu", "down"], ["o"]),      # down: two tiles a pair
    (640, 1152, 5, 1, "f16", True, 700, [], ["qkv", "o", "gu", "down"]),
    (1024, 3072, 8, 8, "", False, 129, [], ["qkv", "o", "gu", "down"]),
])
def test_both_kinds_of_tiles(hidden, inter, nq, nkv, kv, bias, n, pairs, verify):
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=nq, n_kv_heads=nkv, n_layers=2, vocab=700,
                init_std=1.0 / hidden ** 0.5, qkv_bias=bias, cache_dtype=kv)
    case = build_case("mini-bf16", 6, T=4, plant=0, ctx_len=0, cfg_overrides=over, gain_std=0.1, prefill=False)
    model, _ = gpu_model(case)
    assert [g for g in pairs if tiles(model, g, n) != 0] == []
    assert [g for g in verify if tiles(model, g, n) < 1] == []
    prompt = np.random.default_rng(n).integers(0, case.cfg.vocab, size=n).astype(np.int32)
    cache = gpu_cache(case, n)
    nxt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    B.oos_prefill(model, cache, 0, torch.as_tensor(prompt, device="cuda"), n, nxt)
    torch.cuda.synchronize()
    assert B.oos_last_status(model) == B.OOS_OK
    r = oracle.verify_tree(case.view, case.cache_k64, case.cache_v64, 0, prompt, np.arange(n) - 1)
    for l in range(2):
        for got, want in ((cache.k[l], r["tree_k"][l]), (cache.v[l], r["tree_v"][l])):
            got = to_f64(case.cfg, got)
            assert max_rel_err(got, want) <= TOL["bf16"], l
            # every row by itself: 16-bit values, half a step of 2^-8 .. 2^-9 each, and a
            # first layer's error carried on
            row = np.linalg.norm((got - want).reshape(n, -1), axis=1) / np.linalg.norm(want.reshape(n, -1), axis=1)
            assert row.max() <= 2.0 ** -7, (l, int(row.argmax()), row.max())
    if r["top1"][-1] - r["top2"][-1] > 0.05:
        assert int(nxt.item()) == int(r["argmax"][-1])
