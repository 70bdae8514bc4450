"""Top-k past one merge (expand.cu): runs of 256 keys ranked by counting and
merged 8 at a time, on sets up to the size of a whole neighbourhood, against a
sort of the same keys; ragged last runs and groups, nearly empty sets, k below,
at and above a run's length, ties broken by the code; and a planner's frontiers
of different capacities ranked in one launch."""
import numpy as np
import pytest

import paper_2609_21803_gb300 as P
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, capacity, k", [(255, 256, 256), (257, 257, 257), (2048, 2048, 1), (2049, 2049, 2000),
                                            (16385, 16385, 4096),
                                            (262144, 262144, 64), (262145, 300000, 2048), (420000, 420001, 1024),
                                            (200000, 262145, 4096), (3, 300000, 255), (300, 300000, 300)])
def test_large_sets(n, capacity, k):
    prob = P.Problem([dict(W.push_l4_instance(3), max_segments=6)])
    rng = np.random.default_rng(n + k)
    pick = rng.choice(12 ** 6, n, replace=False)
    seqs = np.stack([pick // 12 ** i % 12 for i in range(6)], 1).astype(np.uint8)
    # an order's code: its length, then a digit (mode + 1) per segment, base 13
    code = 6 + ((seqs.astype(np.uint64) + 1) * np.uint64(13) ** np.arange(1, 7, dtype=np.uint64)).sum(1)
    assert int(code[0]) == P.comet_mode_code(tuple(int(m) for m in seqs[0]))
    cost = (rng.integers(0, max(2, n // 3), n) / 16.0 - 4.0).astype(np.float32)
    cost[rng.random(n) < 0.02] = np.inf
    cost[rng.random(n) < 0.02] = np.nan
    f = P.comet_frontier_create(prob.handle, 0, capacity, min(capacity, 64), k)
    P.comet_frontier_add(f, P.pack_mode_seqs(seqs), n, cost, np.zeros(n, np.float32))
    key = np.where(np.isfinite(cost), cost, np.inf)
    order = np.lexsort((code, key))[:k]
    for _ in range(2):
        codes, merit = P.comet_frontier_best(f, k)
        m = len(order)
        assert np.array_equal(codes[:m], code[order])
        assert np.array_equal(merit[:m], key[order].astype(np.float32))
        assert not codes[m:].any() and np.isinf(merit[m:]).all()
    P.comet_frontier_destroy(f)
    prob.close()


def test_frontiers_of_one_launch_are_ranked_as_alone():
    # capacities around 2,048 keys (one merge below, two above) in one launch,
    # whose passes are as many as the largest needs
    insts = [dict(W.push_l4_instance(i), knots_per_segment=3, max_segments=4) for i in range(3)]
    one = W.sequences_up_to(12, 1)
    seeds = [one, one + [(a, b) for a in range(12) for b in range(12)], one[:1]]
    opts = dict(k=64, batch=670, rounds=3, k_ref=64, ref_iters=20)
    prob = P.Problem(insts, {"max_iters": 5})
    many = P.comet_plan_batch(prob.handle, list(range(3)), seeds, opts)
    for i in range(3):
        n = len(seeds[i])
        alone = P.comet_plan(prob.handle, i, P.pack_mode_seqs(seeds[i], np.full(n, i, np.int32)), n, opts)
        for name in ("evaluations", "best", "best_status"):
            assert many[i][name] == alone[name], (i, name)
    prob.close()
