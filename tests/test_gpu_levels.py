"""Passes over the DAG's levels: launched one by one or, for small levels, in one
cluster; a captured plan always launches them one by one.  And the load's
frontiers of rules with few references (one cluster) and with more (launches)."""
import numpy as np
import pytest

import oracle
from paper_2106_06889_gb300 import binding as B
from tests.test_gpu_primitives import check, deep_grammar
from tests.test_oracle_pins import grammar_from_rules

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.gt_create(0)
    yield c
    B.gt_destroy(c)


@pytest.mark.parametrize("wide", [1, 300, 20_000])
def test_captured_levels(ctx, wide):
    """Weights, per-file weights and rule ends inside a plan, over 61 levels."""
    import torch
    g = deep_grammar(wide)
    gh = B.gt_load_grammar(ctx, g)
    counts = torch.empty(g.num_words, dtype=torch.int64, device="cuda")
    p = B.gt_plan_create(ctx, [(gh, B.GT_Q_WORD_COUNT, 0, counts), (gh, B.GT_Q_TERM_VECTOR, 0, None),
                               (gh, B.GT_Q_SEQUENCE_COUNT, 0, None), (gh, B.GT_Q_SEQUENCE_COUNT, 1, None)])
    want = [(1, "offsets word count", oracle.term_vector(g, 0)), (2, "key count", oracle.sequence_count(g, 0)),
            (3, "file key count", oracle.sequence_count(g, 1))]
    try:
        for _ in range(2):
            counts.fill_(-1)
            B.gt_plan_launch(p)
            for i, fields, values in want:
                for f, v in zip(fields.split(), values):
                    assert np.array_equal(B.plan_result_numpy(p, i, f), v), (i, f)
            assert np.array_equal(counts.cpu().numpy().astype(np.uint64), oracle.word_count(g).astype(np.uint64))
    finally:
        B.gt_plan_destroy(p)
        B.gt_free_grammar(gh)


@pytest.mark.parametrize("n", [1, 40, 300])
@pytest.mark.parametrize("refs", [3, 4, 5, 8])
def test_frontiers(ctx, refs, n):
    """Layers of n rules with refs references to the next layer: on either side of four distinct references per rule."""
    V, depth = 40, 4
    rng = np.random.default_rng(refs * n)
    rules = []
    for l in range(depth):
        for i in range(n):
            nxt = V + 1 + (l + 1) * n
            rules.append([int(rng.integers(V))] + [nxt + (i + k * 3) % n if l + 1 < depth else int(rng.integers(V))
                                                   for k in range(refs)])
    root = [V + 1 + i for i in range(n)] + [1, 2, V + 1]
    g = grammar_from_rules(V, [root] + rules, [0, n // 2, len(root)])
    gh = B.gt_load_grammar(ctx, g)
    try:
        assert B.gt_grammar_info_get(gh)["depth"] == depth + 1
        check(gh, g)
    finally:
        B.gt_free_grammar(gh)
