"""Bottom-up rows of a root long enough (more than 12 * 2^20 symbols) that the
references to rules of up to four words are expanded from the rules' first and
last words, longer ones by walking: rules of 1 to 8 words, some through other
rules; a row of a word and its file in 32 bits, and in two words."""
import numpy as np
import pytest

import oracle
from paper_2106_06889_gb300 import binding as B
from paper_2106_06889_gb300.corpus import Grammar
from tests.test_gpu_primitives import take

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [50_000, 2 ** 25])
def test_long_root(V):
    rng = np.random.default_rng(V)
    n, F, flat = (12 << 20) + 77, 70, 600
    rules = [rng.integers(0, V, 1 + i % 6) for i in range(flat)]  # 1 to 6 words
    # a rule between words: 2 to 8 words
    rules += [np.concatenate([rng.integers(0, V, i % 2), [V + 1 + i % flat], rng.integers(0, V, 1 + i % 2)])
              for i in range(300)]
    root = np.where(rng.random(n) < 0.85, (rng.zipf(1.3, n) - 1) % V, V + 1 + rng.integers(0, len(rules), n))
    root[-1] = V - 1
    cuts = np.sort(rng.integers(0, n + 1, F - 1))
    cuts[3] = cuts[4]  # an empty file
    lens = [n] + [len(r) for r in rules]
    g = Grammar(V, np.concatenate([[0], np.cumsum(lens)]).astype(np.int64),
                np.concatenate([root] + rules).astype(np.int32), np.concatenate([[0], cuts, [n]]).astype(np.int64))
    ctx = B.gt_create(0)
    try:
        gh = B.gt_load_grammar(ctx, g)
        for got, want in zip(take(B.gt_term_vector(gh, 0), "offsets", "word", "count"), oracle.term_vector(g, 0)):
            assert np.array_equal(got, want)
        for got, want in zip(take(B.gt_inverted_index(gh), "offsets", "file"), oracle.inverted_index(g)):
            assert np.array_equal(got, want)
        B.gt_free_grammar(gh)
    finally:
        B.gt_destroy(ctx)
