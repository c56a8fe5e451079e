"""Blocks that read each other's shared memory (the k-splits of a GEMM tile, the key
splits of an attention row block): a block may leave, or reuse what the others
read, only once their reads are complete."""

import os
import re

import numpy as np
import pytest
import torch

from cases import build_case

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_00814_gb300", "csrc")


def test_every_cluster_arrival_releases():
    """A relaxed arrival orders none of the thread's earlier accesses, so a peer
    could leave while a pull from its shared memory is still in flight."""
    arrivals = []
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            arrivals += re.findall(r"barrier\.cluster\.arrive[.\w]*", f.read())
    assert arrivals
    assert all(".release" in a for a in arrivals), arrivals


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")
@pytest.mark.parametrize("T,ctx", [(16, 900), (128, 2500)])
def test_pulled_sums_repeat_bit_for_bit(T, ctx):
    """Steps back to back, the next kernel's blocks taking the places of those that
    leave: every pass gives the same bits."""
    from gpu_util import gpu_cache, gpu_model
    from paper_2608_00814_gb300 import binding as B
    over = dict(hidden=1024, intermediate=2048, n_q_heads=8, n_kv_heads=4, n_layers=3, vocab=700, init_std=1.0 / 32)
    case = build_case("mini-bf16", 4, T=T, plant=0, ctx_len=ctx, cfg_overrides=over, gain_std=0.1, prefill=False)
    model, _ = gpu_model(case)
    cache = gpu_cache(case, ctx + 300)
    tok = torch.as_tensor(np.asarray(case.tokens, np.int32), device="cuda")
    par = torch.as_tensor(np.asarray(case.parent, np.int32), device="cuda")
    prompt = torch.as_tensor((np.arange(300) * 37 % 700).astype(np.int32), device="cuda")

    def bits(n):
        return torch.stack([t[ctx:ctx + n].clone() for t in cache.k + cache.v]).view(torch.int16)

    def verify():
        o = B.tree_verify(model, cache, ctx, tok, par, debug=True)
        return [o.final_hidden.view(torch.int32), bits(T)]

    def prefill():
        nxt = torch.zeros(1, dtype=torch.int32, device="cuda")
        B.oos_prefill(model, cache, ctx, prompt, 300, nxt)
        return [nxt, bits(300)]

    for call in (verify, prefill):
        passes = [call() for _ in range(40)]
        torch.cuda.synchronize()
        assert B.oos_last_status(model) == B.OOS_OK
        for p in passes[1:]:
            for a, b in zip(passes[0], p):
                assert torch.equal(a, b)
