"""Top-k of the evaluated set by counting (expand.cu) against a sort of the
same keys: one-pass and chunked sets, k from 1 to the largest, sets smaller
than k, equal merits (ordered by code), infinite and NaN scores (last)."""
import numpy as np
import pytest

import paper_2609_21803_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, capacity, k", [(1, 1, 1), (31, 33, 32), (33, 40, 64), (1025, 1030, 7), (3000, 7096, 64),
                                            (16384, 16384, 256), (16000, 16385, 31), (20736, 60000, 4096),
                                            (5, 20000, 2000)])
def test_topk_matches_a_sort(n, capacity, k):
    prob = P.Problem([W.push_l4_instance(3)])
    rng = np.random.default_rng(n)
    seqs = W.all_sequences(12, 4)[rng.permutation(20736)[:n]]
    packed = P.pack_mode_seqs(seqs)
    # few distinct values, so that ties are broken by the code
    cost = (rng.integers(0, max(2, n // 3), n) / 16.0 - 4.0).astype(np.float32)
    cost[rng.random(n) < 0.02] = np.inf
    cost[rng.random(n) < 0.02] = np.nan
    f = P.comet_frontier_create(prob.handle, 0, capacity, min(capacity, 64), k)
    P.comet_frontier_add(f, packed, n, cost, np.zeros(n, np.float32))
    for _ in range(2):
        codes, merit = P.comet_frontier_best(f, k)
        key = np.where(np.isfinite(cost), cost, np.inf)
        code = np.array([P.comet_mode_code(tuple(s)) for s in seqs], np.uint64)
        order = np.lexsort((code, key))[:k]
        m = len(order)
        assert np.array_equal(codes[:m], code[order])
        assert np.array_equal(merit[:m], key[order].astype(np.float32))
        assert not codes[m:].any() and np.isinf(merit[m:]).all()
    P.comet_frontier_destroy(f)
    prob.close()
