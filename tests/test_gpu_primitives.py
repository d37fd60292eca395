"""The one-pass primitives (scan, radix sort, run reduction) through the
public calls, at the edges of their tiles: 2,048 values per scan and reduction
tile, 2,048 or 6,144 rows per sort tile, the row count at which the sort
changes its tile, runs that cover whole tiles, and (file, key) rows that fit
one 64-bit sort key and that do not.  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2106_06889_gb300 import binding as B
from paper_2106_06889_gb300.corpus import root_only_grammar, sequitur
from tests.test_oracle_pins import grammar_from_rules

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.gt_create(0)
    yield c
    B.gt_destroy(c)


def take(r, *fields):
    out = [B.result_numpy(r, f) for f in fields]
    B.gt_free_result(r)
    return out


def check(gh, g):
    for order in (0, 1):
        for got, want in zip(take(B.gt_sort(gh, order), "word", "count"), oracle.sort_words(g, order)):
            assert np.array_equal(got, want)
    for got, want in zip(take(B.gt_sequence_count(gh, 0), "key", "count"), oracle.sequence_count(g, 0)):
        assert np.array_equal(got, want)
    for got, want in zip(take(B.gt_sequence_count(gh, 1), "file", "key", "count"), oracle.sequence_count(g, 1)):
        assert np.array_equal(got, want)
    for n in (1, 3):
        for got, want in zip(take(B.gt_ranked_index(gh, n), "offsets", "key", "file", "count"),
                             oracle.ranked_index(g, n)):
            assert np.array_equal(got, want)
    for got, want in zip(take(B.gt_cooccurrence(gh), "key", "count"), oracle.cooccurrence(g)):
        assert np.array_equal(got, want)
    for top in (0, 3):
        for got, want in zip(take(B.gt_term_vector(gh, top), "offsets", "word", "count"), oracle.term_vector(g, top)):
            assert np.array_equal(got, want)
    for got, want in zip(take(B.gt_inverted_index(gh), "offsets", "file"), oracle.inverted_index(g)):
        assert np.array_equal(got, want)


# windows = tokens - 2: 2048 and 4096 rows and one more or less, several tiles, one row
EDGES = [3, 2049, 2050, 2051, 4097, 4098, 4099, 8194, 20_483]


@pytest.mark.parametrize("n", EDGES)
@pytest.mark.parametrize("text", ["one_word", "few", "distinct"])
def test_tile_edges(ctx, n, text):
    """One file, no rules: one key whose run covers every tile, a few long runs, all keys distinct."""
    rng = np.random.default_rng(n)
    V = {"one_word": 2, "few": 5, "distinct": 30_011}[text]
    toks = {"one_word": np.ones(n), "few": rng.integers(0, V, n), "distinct": np.arange(n) * 7 % V}[text].astype(np.int32)
    g = root_only_grammar(toks, [n], V)
    gh = B.gt_load_grammar(ctx, g)
    try:
        check(gh, g)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("strategy", [1, 2])
@pytest.mark.parametrize("V,F", [(2 ** 21, 3), (2 ** 20, 17), (2 ** 20, 15), (70_000, 64)])
def test_file_keys(ctx, V, F, strategy):
    """(file, 3-word key) rows of 64 bits and more, of 63 bits and of fewer, top-down and
    bottom-up (by the global sort), empty files among them."""
    rng = np.random.default_rng(V + F)
    toks = (rng.zipf(1.3, 9000) % V).astype(np.int32)
    toks[1000:2000] = toks[4000:5000]  # a repeated passage: rules
    toks[-1] = V - 1
    cuts = np.sort(rng.integers(0, toks.shape[0] + 1, F - 1))
    cuts[F // 2:F // 2 + 1] = cuts[F // 2 - 1]  # an empty file
    lens = np.diff(np.concatenate([[0], cuts, [toks.shape[0]]]))
    g = sequitur(toks, lens, V)
    B.gt_set_param(ctx, "file_strategy", strategy)
    B.gt_set_param(ctx, "bu_local", 0)
    gh = B.gt_load_grammar(ctx, g)
    try:
        check(gh, g)
    finally:
        B.gt_free_grammar(gh)
        B.gt_set_param(ctx, "file_strategy", 0)
        B.gt_set_param(ctx, "bu_local", 1)


@pytest.mark.parametrize("n", [2 ** 20 - 1 + 2, 2 ** 20 + 2, 171 * 6144 + 2, 171 * 6144 + 3])
def test_sort_tile_change(ctx, n):
    """Rows just below and above 2^20, where the sort goes from 2,048- to 6,144-row tiles, and at
    the edge of a large tile."""
    rng = np.random.default_rng(n)
    toks = (rng.zipf(1.2, n) % 5000).astype(np.int32)
    g = root_only_grammar(toks, [n // 2, n - n // 2], 5000)
    gh = B.gt_load_grammar(ctx, g)
    try:
        for per_file, fields in ((0, ("key", "count")), (1, ("file", "key", "count"))):
            for got, want in zip(take(B.gt_sequence_count(gh, per_file), *fields), oracle.sequence_count(g, per_file)):
                assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("V", [45, 70_000])
@pytest.mark.parametrize("F", [1, 31, 32, 33, 64])
def test_file_sets(ctx, F, V):
    """Inverted index: words in few files and in most of them, one and two 32-file halves."""
    rng = np.random.default_rng(F * V)
    toks = (rng.zipf(1.2, 6000) % V).astype(np.int32)
    cuts = np.sort(rng.integers(0, toks.shape[0] + 1, F - 1))
    g = root_only_grammar(toks, np.diff(np.concatenate([[0], cuts, [toks.shape[0]]])), V)
    gh = B.gt_load_grammar(ctx, g)
    try:
        for got, want in zip(take(B.gt_inverted_index(gh), "offsets", "file"), oracle.inverted_index(g)):
            assert np.array_equal(got, want)
        # the same tolerance as the TF-IDF test: one quotient, logarithm (1 ulp) and product in float64
        for got, want in zip(take(B.gt_tfidf(gh), "offsets", "word", "tfidf"), oracle.tfidf(g)):
            assert np.allclose(got, want, rtol=1e-15, atol=0)
    finally:
        B.gt_free_grammar(gh)


def deep_grammar(wide):
    """A chain of 60 rules (rule r holds a word and rule r + 1), each also used by the root's two
    files, over ``wide`` rules of two words on one level: with wide = 20,000 that level is too large
    to share a launch with the small ones."""
    V, depth = 50, 60
    rng = np.random.default_rng(wide)
    chain = [[int(rng.integers(V)), V + r + 1] if r < depth else [3, 4] for r in range(1, depth + 1)]
    flat = [[int(a), int(b)] for a, b in rng.integers(0, V, (wide, 2))]
    users = [[V + depth + 1 + i, V + depth + 1 + (i * 7) % wide, int(rng.integers(V))] for i in range(wide)]
    first = V + depth + 1 + wide
    root = [V + 1, 5, V + 30, V + 1] + [first + i for i in range(wide)] + [V + r for r in range(1, depth + 1)]
    return grammar_from_rules(V, [root] + chain + flat + users, [0, 3 + wide // 3, len(root)])


@pytest.mark.parametrize("wide", [1, 300, 20_000])
def test_levels(ctx, wide):
    """Level passes (weights, per-file weights, head/tail buffers) over many small levels, alone
    and after a level too large for them; head/tail into buffers that are not 8-byte aligned."""
    import torch
    g = deep_grammar(wide)
    gh = B.gt_load_grammar(ctx, g)
    try:
        w = torch.empty(g.num_rules, dtype=torch.int64, device="cuda")
        B.gt_rule_weights(gh, w)
        assert np.array_equal(w.cpu().numpy().astype(np.uint64), oracle.rule_weights(g))
        raw = [torch.full((2 * g.num_rules + 2,), -7, dtype=torch.int32, device="cuda") for _ in range(2)]
        for shift in (0, 1):
            views = [x[shift:shift + 2 * g.num_rules] for x in raw]
            B.gt_head_tail(gh, *views)
            for got, want in zip(views, oracle.head_tail(g)):
                assert np.array_equal(got.cpu().numpy().reshape(-1, 2), np.asarray(want).reshape(-1, 2))
        check(gh, g)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("V", [6, 70_000, 200_000])
@pytest.mark.parametrize("F", [65, 300, 700])
def test_ranked_runs(ctx, F, V):
    """Ranked index of many files, keys in 1 to all of them (put in order by a thread, a warp or a
    CTA): (key, file) in one word for the two smaller vocabularies, by the expanded files otherwise;
    files of 0 to 2 words among them, repeated passages (rules) in some."""
    rng = np.random.default_rng(F + V)
    lens = rng.integers(0, 60, F)
    lens[:4] = [0, 1, 2, 3]
    n = int(lens.sum())
    toks = np.where(rng.random(n) < 0.9, rng.integers(0, 3, n), rng.integers(0, V, n)).astype(np.int32)
    g = sequitur(toks, lens, V)
    gh = B.gt_load_grammar(ctx, g)
    try:
        for k in (1, 3):
            for got, want in zip(take(B.gt_ranked_index(gh, k), "offsets", "key", "file", "count"),
                                 oracle.ranked_index(g, k)):
                assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("V", [50, 2 ** 20, 2 ** 20 + 1])
@pytest.mark.parametrize("w", [1, 3, 4, 192, 255, 256, 0xfff3, (1 << 20) + 0xabcde])
@pytest.mark.parametrize("long_root", [True, False])
def test_weight_components(ctx, w, V, long_root):
    """3-word rows whose weight is part of the key's word (vocabularies up to 2^20, at most three
    tokens per window: the long root) and beside it: a rule x x x of weight w, used by doubling rules,
    x the largest word, so that all bits of the key are set where V is a power of two."""
    x, top = V - 1, w.bit_length() - 1
    rules = [[x, x, x]] + [[V + k, V + k] for k in range(1, top + 1)]  # rule k + 1 = 2^k times x x x
    uses = [V + 1 + k for k in range(top + 1) if (w >> k) & 1]
    rng = np.random.default_rng(w)
    n = 100 + (2 * w if long_root else 0)
    root = rng.integers(0, V, n).tolist()
    for i, u in enumerate(uses):
        root.insert(3 * i + 1, u)
    g = grammar_from_rules(V, [root] + rules, [0, 40, len(root)])
    gh = B.gt_load_grammar(ctx, g)
    try:
        for got, want in zip(take(B.gt_sequence_count(gh, 0), "key", "count"), oracle.sequence_count(g, 0)):
            assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("F,V,per_file", [(65, 6, 50), (300, 70_000, 50), (2_000, 200_000, 50), (2_100, 2_000_000, 50),
                                          (300, 70_000, 16_000), (70, 2 ** 25, 60_000)])
def test_word_rows(ctx, F, V, per_file):
    """Term vectors and inverted index of more than 64 files from the expanded files: a row of a word
    and its file in 32 bits, or (the last) in two words; one file that expands past a tile's stage
    from few symbols, files of 0 and 1 words; the two largest have a root of more than 2^20 symbols,
    whose references to short rules are expanded from the rules' ends."""
    rng = np.random.default_rng(F + V)
    lens = rng.integers(0, per_file, F)
    lens[:3] = [0, 1, 9000]
    n = int(lens.sum())
    toks = np.where(rng.random(n) < 0.7, rng.integers(0, 5, n), rng.integers(0, V, n)).astype(np.int32)
    toks[1:9001] = np.tile(toks[1:10], 1000)
    toks[-1] = V - 1
    g = sequitur(toks, lens, V)
    gh = B.gt_load_grammar(ctx, g)
    try:
        tv, ii = B.gt_run_batch(ctx, [(gh, B.GT_Q_TERM_VECTOR, 0, None), (gh, B.GT_Q_INVERTED_INDEX, 0, None)])
        for got, want in zip(take(tv, "offsets", "word", "count"), oracle.term_vector(g, 0)):
            assert np.array_equal(got, want)
        for got, want in zip(take(ii, "offsets", "file"), oracle.inverted_index(g)):
            assert np.array_equal(got, want)
        for got, want in zip(take(B.gt_term_vector(gh, 2), "offsets", "word", "count"), oracle.term_vector(g, 2)):
            assert np.array_equal(got, want)
    finally:
        B.gt_free_grammar(gh)
