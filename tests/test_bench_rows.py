"""Bytes that bench.py credits to the 3-word count's kernels: rows of one word
(vocabularies up to 2^20, at most three tokens per window), else key and weight."""
import sys
from pathlib import Path

import pytest

sys.path.insert(0, str(Path(__file__).resolve().parent.parent))
import bench  # noqa: E402


@pytest.mark.parametrize("V,tokens,one_word", [(500_000, 3300, True), (500_000, 3301, False), (1 << 20, 1200, True),
                                               ((1 << 20) + 1, 1200, False)])
def test_rows_of_one_word(V, tokens, one_word):
    info = {"num_syms": 1000, "num_words": V, "owned_windows": 1100, "num_tokens": tokens}
    kb = bench.kernel_bytes("nested_500m", info, {"distinct_3grams": 700, "root_len": 400})
    assert kb["radix_pass"] == (("radix_downsweep_kernel<0>", 16 * 1100) if one_word
                                else ("radix_downsweep_kernel<4>", 24 * 1100))
    assert kb["seq_reduce"][1] == (8 if one_word else 12) * 1100 + 16 * 700
