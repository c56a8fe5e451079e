"""Common tokens in the hint bank: the last committed token, and longer pieces of the
suffix, in every chunk and across the ends of lanes, halves, chunks and of the bank."""

import numpy as np
import pytest

from test_gpu_hint import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5, 127, 128, 129, 255, 256, 257, 300, 511, 512, 1000, 4097, 70_001])
@pytest.mark.parametrize("vocab", [2, 3, 20])
@pytest.mark.parametrize("shift", [0, 1])
def test_common_tokens(n, vocab, shift):
    rng = np.random.default_rng(1000 * n + 10 * vocab + shift)
    bank = rng.integers(0, vocab, size=n).tolist()
    for eos in (0, vocab - 1, 99):                    # a token of the bank, or of no bank
        for m in (1, 2, 3, 7, 12):                    # the suffix: one token to more than are tried
            y = rng.integers(0, vocab, size=m).tolist()
            _check(bank, eos, y, [[1, 2, 3]], 5, 6, 24, shift)


@pytest.mark.parametrize("n", [(1 << 20) + 3, 1_300_000])
def test_common_tokens_of_a_large_bank(n):
    """Past what packing reads without span maxima: 5 % of the bank is the last
    token, a few places hold longer pieces of the suffix, one of them the bank's end."""
    rng = np.random.default_rng(n)
    bank = rng.integers(100, 50000, size=n)
    bank[rng.random(n) < 0.05] = 7
    y = [5, 6, 8, 9, 7]
    for at in (254, 511, 127 + 256 * 1000, n // 2, n - 9):
        bank[at:at + 4] = y[1:]
    r = _check(bank.tolist(), 1, y, [], 8, 5, 40)
    assert r["match_n"] == 4 and r["hint_lanes"] == 5
    bank[n - 5:] = y                                   # nothing follows it: does not count
    assert _check(bank.tolist(), 1, y, [], 8, 5, 40)["match_n"] == 4


@pytest.mark.parametrize("length", range(1, 8))
@pytest.mark.parametrize("at", [0, 1, 3, 120, 125, 127, 128, 130, 250, 254, 255, 256, 258, 505])
def test_every_length_at_every_edge(length, at):
    """One occurrence of the suffix's last `length` tokens, ending inside a chunk or
    just past one's start, at every way of lying across lanes and halves."""
    rng = np.random.default_rng(at)
    bank = rng.integers(100, 5000, size=600).tolist()
    y = [11, 12, 13, 14, 15, 16, 17]
    bank[at:at + length] = y[7 - length:]
    r = _check(bank, 1, y, [], 3, 4, 16)
    assert r["match_n"] == length and r["hint_lanes"] == 1
