"""Radix sort forms that the smaller primitive tests do not reach: tiles of 8192
keys without values (from 2^22 rows on; 64-bit rows of the 3-word count, 32-bit
rows of a word and its file), and 64-bit look-back words ("radix_wide", taken by
itself from 2^30 rows on).  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2106_06889_gb300 import binding as B
from paper_2106_06889_gb300.corpus import root_only_grammar, sequitur
from tests.test_gpu_primitives import check, take

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.gt_create(0)
    yield c
    B.gt_destroy(c)


ROWS = [(1 << 22) - 1, 1 << 22, (1 << 22) + 1, 513 * 8192 - 1, 513 * 8192, 513 * 8192 + 1]


@pytest.mark.parametrize("n", ROWS)
def test_key_only_tiles_64(ctx, n):
    """One-word rows of the 3-word count: n windows, sorted with room for one more."""
    rng = np.random.default_rng(n)
    toks = (rng.zipf(1.2, n + 2) % 4000).astype(np.int32)
    g = root_only_grammar(toks, [n + 2], 4000)
    gh = B.gt_load_grammar(ctx, g)
    try:
        for got, want in zip(take(B.gt_sequence_count(gh, 0), "key", "count"), oracle.sequence_count(g, 0)):
            assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("n", ROWS)
def test_key_only_tiles_32(ctx, n):
    """Rows of a word and its file in 32 bits: n words in 70 files."""
    rng = np.random.default_rng(n)
    toks = (rng.zipf(1.2, n) % 3000).astype(np.int32)
    cuts = np.sort(rng.integers(0, n + 1, 69))
    g = root_only_grammar(toks, np.diff(np.concatenate([[0], cuts, [n]])), 3000)
    gh = B.gt_load_grammar(ctx, g)
    try:
        for got, want in zip(take(B.gt_inverted_index(gh), "offsets", "file"), oracle.inverted_index(g)):
            assert np.array_equal(got, want)
        for got, want in zip(take(B.gt_term_vector(gh, 0), "offsets", "word", "count"), oracle.term_vector(g, 0)):
            assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("n,V,F", [(20_483, 5000, 5), (40_000, 2 ** 21, 9), (60_000, 70_000, 80), (60_000, 2 ** 20 + 1, 300)])
def test_wide_look_back_words(ctx, n, V, F):
    """Every sort of the engine, keys of 32 and 64 bits, with values of 0, 4 and 8 bytes, over several tiles."""
    rng = np.random.default_rng(n + V)
    toks = (rng.zipf(1.2, n) % V).astype(np.int32)
    toks[1000:3000] = toks[7000:9000]
    toks[-1] = V - 1
    cuts = np.sort(rng.integers(0, n + 1, F - 1))
    g = sequitur(toks, np.diff(np.concatenate([[0], cuts, [n]])), V)
    B.gt_set_param(ctx, "radix_wide", 1)
    B.gt_set_param(ctx, "bu_local", 0)
    gh = B.gt_load_grammar(ctx, g)
    try:
        check(gh, g)
    finally:
        B.gt_free_grammar(gh)
        B.gt_set_param(ctx, "radix_wide", 0)
        B.gt_set_param(ctx, "bu_local", 1)
