"""The failure path of the waits in pairs of CTAs and in prefill, exercised without a
fault: with a wait limit of one nanosecond the kernels give up, drain their copies and
MMAs, free their tensor memory and return; the call reports it; and the handle, with
the default limit again, gives what a fresh one gives.  Collected near the end."""

import numpy as np
import pytest
import torch

from cases import build_case
from gpu_util import gpu_cache, gpu_model

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2608_00814_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("hidden,inter,T,n", [
    (128, 11520, 128, 0),    # gate/up of a tree in pairs
    (256, 512, 128, 0),      # in tiles of 64 tokens
    (256, 512, 0, 300),      # a prefill chunk in token tiles
    (2432, 3072, 0, 1280),   # in pairs' tiles
    (256, 512, 0, 2100),     # a chunk, then a tree
])
def test_limit_runs_out_and_the_handle_recovers(hidden, inter, T, n):
    over = dict(hidden=hidden, intermediate=inter, n_q_heads=15, n_kv_heads=5, n_layers=2, vocab=700,
                init_std=1.0 / hidden ** 0.5)
    m = T or n
    case = build_case("mini-bf16", 2, T=T or 4, plant=0, ctx_len=40, cfg_overrides=over, prefill=False)
    model, w = gpu_model(case)
    tok = torch.as_tensor(np.random.default_rng(m).integers(0, 700, size=m).astype(np.int32), device="cuda")
    par = torch.arange(m, dtype=torch.int32, device="cuda") - 1

    def call(model):
        cache = gpu_cache(case, 40 + m)
        if T:
            o = B.tree_verify(model, cache, 40, tok, par)
            out = [o.accepted_len, o.bonus]
        else:
            out = [torch.full((1,), -1, dtype=torch.int32, device="cuda")]
            B.oos_prefill(model, cache, 40, tok, n, out[0])
        torch.cuda.synchronize()   # the kernels returned
        return [t.view(torch.int16) for t in cache.k + cache.v] + out, B.oos_last_status(model)

    B.oos_set_wait_limit(model, 1)
    out, status = call(model)
    assert status == B.OOS_ETIMEOUT
    if T:
        assert int(out[-2]) == 0 and int(out[-1]) == -1
    B.oos_set_wait_limit(model, 0)
    again, status = call(model)
    assert status == B.OOS_OK
    fresh, status = call(B.OosModel(case.cfg, w))
    assert status == B.OOS_OK
    for a, b in zip(again, fresh):
        assert torch.equal(a, b)
