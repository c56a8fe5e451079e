"""The allocation-free LM-head argmax (oos_lm_head_argmax_static), through
the C ABI, against the CPU checker's LM head and against the LM head of
oos_tree_verify_debug on the same rows.

The entry point is for callers that cannot allocate device memory (inside a
CUDA graph that someone else is capturing, under a memory pool they do not
own, with a locked allocator): its scratch is a fixed device array inside the
library that every call shares.  So it is called twice in a row, to check
that the second call starts from a clean state.  The file is collected last on
purpose: it shares nothing with the other tests and must pass both alone in a
fresh process and after them.
"""

import numpy as np
import pytest
import torch

import oracle
from cases import build_case
from gpu_util import GATE, TOL, gpu_cache, gpu_model, max_rel_err, run

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2608_00814_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("name,T", [("tiny", 8), ("mini-bf16", 16), ("mini-bf16", 128)])
def test_static_argmax_matches_oracle_and_verify(name, T):
    case = build_case(name, 0, T=T, plant=3, recipe=dict(kind="uniform", max_depth=6))
    model, w = gpu_model(case)
    kv = gpu_cache(case, case.ctx_len + T)
    g = run(model, kv, case.ctx_len, case.tokens, case.parent)
    hidden = g["debug_outs"].final_hidden     # fp32 [T, H] final-RMSNorm rows from the verify
    # the checker's LM head on the very same rows, in fp64 over the same weights
    ref_arg, ref_t1, ref_t2 = oracle.lm_head_argmax(case.view, hidden.cpu().numpy().astype(np.float64))
    ref_margin = ref_t1 - ref_t2
    dtype = B.OOS_DTYPE_BF16 if case.cfg.dtype == "bf16" else B.OOS_DTYPE_F32
    tol_v, gate_v = TOL[case.cfg.dtype], GATE[case.cfg.dtype]
    for call in range(2):
        arg = torch.full((T,), -7, dtype=torch.int32, device="cuda")
        t1 = torch.full((T,), float("nan"), dtype=torch.float32, device="cuda")
        t2 = torch.full((T,), float("nan"), dtype=torch.float32, device="cuda")
        B.oos_lm_head_argmax_static(dtype, case.cfg.vocab, case.cfg.hidden, w["lm_head"], hidden, T, arg, t1, t2)
        torch.cuda.synchronize()
        a = arg.cpu().numpy()
        v1 = t1.cpu().numpy().astype(np.float64)
        v2 = t2.cpu().numpy().astype(np.float64)
        # vs the checker: fp32 dot products of fp32 rows, so the fp32 tolerance and gate
        assert max_rel_err(v1, ref_t1) <= TOL["f32"], (call, max_rel_err(v1, ref_t1))
        assert max_rel_err(v2, ref_t2) <= TOL["f32"], (call, max_rel_err(v2, ref_t2))
        sep = ref_margin > GATE["f32"]
        assert np.array_equal(a[sep], ref_arg[sep]), call
        assert sep.sum() >= T // 2
        # vs the existing entry point (the verify's fused LM head), at the tolerance of its dtype
        assert max_rel_err(v1, g["top1"].astype(np.float64)) <= tol_v
        assert max_rel_err(v2, g["top2"].astype(np.float64)) <= tol_v
        sep_v = g["top1"] - g["top2"] > gate_v
        assert np.array_equal(a[sep_v], g["argmax"][sep_v]), call


def test_static_argmax_rejects_oversized_T():
    x = torch.zeros(1, dtype=torch.float32, device="cuda")   # never read: the call is rejected first
    i = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(B.OosError) as e:
        B.oos_lm_head_argmax_static(B.OOS_DTYPE_F32, 16, 4, x, x, 129, i, x, x)
    assert e.value.code == B.OOS_EINVAL


@pytest.mark.parametrize("vocab,hidden,T,bf16,shift", [
    (1, 8, 1, True, 0), (700, 1000, 3, True, 0), (701, 1000, 17, True, 0),   # row groups cut by the matrix end
    (300, 24, 128, True, 0), (301, 24, 128, False, 0),                       # every token group size in use
    (500, 1001, 9, True, 0), (500, 64, 9, True, 1), (333, 64, 33, False, 1),  # no 16-byte rows: element by element
])
def test_static_argmax_shapes(vocab, hidden, T, bf16, shift):
    """Sizes at the edges of the kernel's row and token groups, and rows that
    16-byte loads cannot read, against fp64 products of the same numbers."""
    g = torch.Generator().manual_seed(vocab + T)
    dt = torch.bfloat16 if bf16 else torch.float32
    w = torch.randn(vocab * hidden + shift, generator=g).to(dt).cuda()[shift:].view(vocab, hidden)
    h = torch.randn(T * hidden + shift, generator=g).cuda()[shift:].view(T, hidden)
    arg = torch.full((T,), -7, dtype=torch.int32, device="cuda")
    t1, t2 = torch.zeros(T, device="cuda"), torch.zeros(T, device="cuda")
    B.oos_lm_head_argmax_static(B.OOS_DTYPE_BF16 if bf16 else B.OOS_DTYPE_F32, vocab, hidden, w, h, T, arg, t1, t2)
    lg = h.cpu().double() @ w.cpu().double().T
    top = lg.topk(min(2, vocab), -1)
    # fp32 products and sums: 2^-24 a step over chains of hidden/32 and a tree, on
    # sums of size sqrt(hidden)
    tol = 2.0 ** -24 * (hidden / 32 + 16) * hidden ** 0.5 * 4
    assert (t1.cpu().double() - top.values[:, 0]).abs().max() <= tol
    if vocab > 1:
        assert (t2.cpu().double() - top.values[:, 1]).abs().max() <= tol
        sure = top.values[:, 0] - top.values[:, 1] > 2 * tol
        assert torch.equal(arg.cpu()[sure], top.indices[:, 0][sure].int())
    else:
        assert int(arg[0]) == 0 and torch.isinf(t2).all()
