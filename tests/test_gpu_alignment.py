"""Norm gains and biases on 8-byte boundaries: every entry point reads them so."""

import numpy as np
import pytest
import torch

from cases import build_case
from gpu_util import gpu_cache, gpu_model

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2608_00814_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("hidden,inter,n", [
    (1280, 3072, 2048),   # q/k/v and gate/up in pairs' tiles
    (2432, 4096, 1700),   # down in pairs' tiles
    (256, 512, 300),      # token tiles
    (256, 512, 100),      # a tree
])
def test_vectors_off_16_byte_boundaries(hidden, inter, n):
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=16, n_kv_heads=8, n_layers=2, vocab=700,
                init_std=1.0 / hidden ** 0.5, qkv_bias=True, qk_norm=True)
    case = build_case("mini-bf16", 4, T=4, plant=0, ctx_len=0, cfg_overrides=over, gain_std=0.1, prefill=False)
    _, w = gpu_model(case)

    def shifted(t):
        u = torch.empty(t.numel() + 4, dtype=t.dtype, device="cuda")[4:]
        assert u.data_ptr() % 16 == 8
        return u.copy_(t)

    off = dict(w, final_norm=shifted(w["final_norm"]), layers=[
        {k: shifted(t) if t is not None and t.dim() == 1 else t for k, t in L.items()} for L in w["layers"]])
    tok = torch.as_tensor(np.random.default_rng(n).integers(0, 700, size=n).astype(np.int32), device="cuda")
    kv = []
    for weights in (w, off):
        model, cache = B.OosModel(case.cfg, weights), gpu_cache(case, n)
        nxt = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        B.oos_prefill(model, cache, 0, tok, n, nxt)
        assert B.oos_last_status(model) == B.OOS_OK
        kv.append([t.view(torch.int16).clone() for t in cache.k + cache.v] + [nxt])
    for a, b in zip(*kv):
        assert torch.equal(a, b)
