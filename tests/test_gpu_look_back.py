"""Look-backs of the primitives (scan, radix sort, run reduction, root
expansion) whose wait runs out: the tile waited for is counted from its input,
so the load and every analytic stay equal to the oracle.  "look_back_polls" 0
makes each look-back count any tile that it does not find published at its
first read; the sizes take several tiles of every primitive."""
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
    B.gt_set_param(c, "look_back_polls", 0)
    B.gt_set_param(c, "bu_local", 0)
    yield c
    B.gt_destroy(c)


def text(n, V, F, seed):
    rng = np.random.default_rng(seed)
    toks = (rng.zipf(1.2, n) % V).astype(np.int32)
    for a in rng.integers(0, n - 4000, 20):  # repeated passages: rules
        b = int(rng.integers(0, n - 4000))
        toks[a:a + 2000] = toks[b:b + 2000]
    toks[-1] = V - 1
    cuts = np.sort(rng.integers(0, n + 1, F - 1))
    return toks, np.diff(np.concatenate([[0], cuts, [n]])), V


@pytest.mark.parametrize("polls", [0, 1, 1 << 22])
@pytest.mark.parametrize("n,V,F", [(150_001, 5000, 5), (120_000, 2 ** 21, 9), (150_000, 70_000, 80),
                                   (150_000, 2 ** 20 + 1, 300)])
def test_missing_tiles_are_counted(ctx, n, V, F, polls):
    """Top-down and bottom-up, rows of one word and of two, the structure that a load keeps."""
    g = sequitur(*text(n, V, F, n + F))
    B.gt_set_param(ctx, "look_back_polls", polls)
    gh = B.gt_load_grammar(ctx, g)
    try:
        check(gh, g)
        B.gt_set_param(ctx, "seq_path", 2)
        for got, want in zip(take(B.gt_sequence_count(gh, 0), "key", "count"), oracle.sequence_count(g, 0)):
            assert np.array_equal(got, want)
    finally:
        B.gt_set_param(ctx, "seq_path", 1)
        B.gt_set_param(ctx, "look_back_polls", 0)
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("text_of", ["one_word", "distinct"])
def test_runs_over_missing_tiles(ctx, text_of):
    """One run over every tile, and a head in every row; tiles of 6144 rows in the sort."""
    n, V = (1 << 20) + 5000, 1 << 21
    toks = (np.ones(n) if text_of == "one_word" else np.arange(n)).astype(np.int32)
    g = root_only_grammar(toks, [n // 3, n - n // 3], V)
    gh = B.gt_load_grammar(ctx, g)
    try:
        for per_file, fields in ((0, ("key", "count")), (1, ("file", "key", "count"))):
            for got, want in zip(take(B.gt_sequence_count(gh, per_file), *fields), oracle.sequence_count(g, per_file)):
                assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)


def test_poll_limits(ctx):
    for bad in (-1, (1 << 22) + 1):
        with pytest.raises(B.GtError):
            B.gt_set_param(ctx, "look_back_polls", bad)
