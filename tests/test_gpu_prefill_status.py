"""A bad token anywhere in a prompt is reported, however the prompt is cut into
chunks, and the next call starts from a clean status."""

import pytest
import torch

from cases import build_case
from gpu_util import gpu_cache, gpu_model

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2608_00814_gb300 import binding as B  # noqa: E402


@pytest.mark.parametrize("name,max_T,n,spots", [
    ("mini-bf16", 128, 2049, (7, 2047, 2048)),        # a wide chunk, then one token as a tree
    ("mini-bf16", 16, 2176, (7, 2100)),               # then 128 tokens as a tree
    ("mini-bf16", 128, 4096 + 5, (7, 2050, 4098)),
    ("tiny", 16, 40, (3, 20, 39)),                    # fp32: trees of max_T tokens
])
def test_a_bad_token_of_any_chunk_is_reported(name, max_T, n, spots):
    case = build_case(name, 5, T=4, plant=0, ctx_len=0, prefill=False)
    model, _ = gpu_model(case, max_T=max_T)
    cache = gpu_cache(case, n)
    tok = torch.zeros(n, dtype=torch.int32, device="cuda")
    for at in spots:
        for bad in (case.cfg.vocab, -1):
            tok[at] = bad
            B.oos_prefill(model, cache, 0, tok, n, None)
            assert B.oos_last_status(model) == B.OOS_ETREE, (at, bad)
            tok[at] = 0
        B.oos_prefill(model, cache, 0, tok, n, None)
        assert B.oos_last_status(model) == B.OOS_OK, at
