"""oos_lm_head_argmax_static with rows so long that a row group's element offsets pass
2^32.  Collected last, as the other test of this entry point."""

import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2608_00814_gb300 import binding as B  # noqa: E402


def test_row_group_past_32_bit_offsets():
    vocab, hidden = 8, 640_000_000     # row 7 starts 4.48e9 elements in
    w = torch.zeros(vocab, hidden, dtype=torch.bfloat16, device="cuda")
    h = torch.zeros(1, hidden, dtype=torch.float32, device="cuda")
    w[7, hidden - 5], w[3, hidden - 5] = 2.0, 1.0
    h[0, hidden - 5] = 3.0
    arg = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    t1, t2 = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    B.oos_lm_head_argmax_static(B.OOS_DTYPE_BF16, vocab, hidden, w, h, 1, arg, t1, t2)
    assert (int(arg), float(t1), float(t2)) == (7, 6.0, 3.0)
