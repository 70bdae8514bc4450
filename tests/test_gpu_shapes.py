"""Launch shapes and horizon edges of the evaluators: results do not depend on
how many TOs share a launch (CTA size, start order, warps in step) nor on what
other problems are alive, and the bimanual kernel's stage loops (a thread per
stage, two stages per warp, copy rings) hold at horizons around their strides.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TIMING = {"h_min": 0.05, "h_max": 0.2, "T_max": 100.0}


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_21803_gb300 import build as B
    B.build()
    import paper_2609_21803_gb300 as P
    P.lib()
    torch.cuda.set_device(0)
    return P


def _dev(P, seqs, idx=None):
    packed = P.pack_mode_seqs(seqs, idx)
    return torch.from_numpy(packed.view(np.uint8).reshape(len(seqs), P.MODE_SEQ_BYTES)).cuda()


def _run(P, prob, d, timed, max_iters):
    """Cost, trajectory bits and status of one launch."""
    n = d.shape[0]
    stride = 9 * ((prob.stride - 4) // 7) + 5 if timed else prob.stride
    cost, viol = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    st, iters = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    traj = torch.zeros(n, stride, device="cuda")
    if timed:
        P.comet_eval_modes_timed(prob.handle, TIMING, d, n, None, max_iters, cost, traj, st)
    else:
        P.comet_eval_modes_budget(prob.handle, d, n, None, max_iters, cost, traj, st)
    P.comet_eval_stats(prob.handle, viol, None, iters, None)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in (cost, viol, st, iters, traj)]


def _l(inst, K, L):
    return dict(inst, knots_per_segment=K, max_segments=L)


@pytest.mark.parametrize("timed", [False, True])
@pytest.mark.parametrize("K,L", [(9, 1), (11, 3), (20, 4)])
def test_results_do_not_depend_on_the_launch_size(P, timed, K, L):
    # 5 orders alone (a CTA each past N = 32, out of step) and the same ones
    # tiled to launches of the resident warps (four a CTA, out of step) and of
    # one and a half times as many (in step);
    # instances of two segment lengths, so that the longest start first
    insts = [_l(W.push_l4_instance(0), K, L), _l(W.push_l4_instance(1), K + 1, L)]
    rng = np.random.default_rng(3)
    seqs = [tuple(int(m) for m in rng.integers(0, 12, rng.integers(1, L + 1))) for _ in range(5)]
    idx = np.array([0, 1, 0, 1, 1], np.int32)
    prob = P.Problem(insts)
    c = P.comet_get_launch_config(prob.handle)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    resident = sms * c["blocks_per_sm"] * c["warps_per_block"]
    few = _run(P, prob, _dev(P, seqs, idx), timed, 60)
    for tiles in (resident // 5 + 1, resident * 3 // 10 + 1):
        many = _run(P, prob, _dev(P, seqs * tiles, np.tile(idx, tiles)), timed, 60)
        for a, b in zip(few, many):
            b = b.reshape((tiles,) + a.shape)
            assert (b.view(np.int32) == a.view(np.int32)[None]).all()
    prob.close()


@pytest.mark.parametrize("task", ["push", "timed", "bimanual"])
def test_a_smaller_problem_made_later_leaves_a_larger_one_usable(P, task):
    if task == "bimanual":
        big, small, n_modes = _l(W.bimanual_instance(0), 30, 6), _l(W.bimanual_instance(0), 3, 1), 507
    else:
        big, small, n_modes = _l(W.push_l4_instance(0), 100, 4), _l(W.push_l4_instance(0), 4, 1), 12
    rng = np.random.default_rng(4)
    L = big["max_segments"]
    d = _dev(P, [tuple(int(m) for m in rng.integers(0, n_modes, L)) for _ in range(3)])
    d1 = _dev(P, [(1,), (2,)])
    a = P.Problem([big])
    first = _run(P, a, d, task == "timed", 4)
    b = P.Problem([small])
    _run(P, b, d1, task == "timed", 4)
    again = _run(P, a, d, task == "timed", 4)
    for x, y in zip(first, again):
        np.testing.assert_array_equal(x.view(np.int32), y.view(np.int32))
    a.close()
    b.close()


@pytest.mark.parametrize("K,L", [(1, 1), (2, 1), (3, 1), (4, 1), (5, 1), (8, 1), (9, 1), (13, 1), (17, 2), (64, 2),
                                 (43, 3), (60, 3)])
def test_bimanual_first_iterate_at_horizon_edges(P, K, L):
    # the bar of one FP32 iteration against FP64 is 1e-4 of the largest entry
    # at 15 stages; the sweep and the forward chain add up stage by stage, so
    # it grows with N / 15
    N = K * L
    inst = _l(W.bimanual_instance(5), K, L)
    rng = np.random.default_rng(100 + N)
    n = 8
    seqs = [tuple(int(m) for m in rng.integers(0, 507, L)) for _ in range(n)]
    prob = P.Problem([inst])
    r = prob.eval(_dev(P, seqs), want_traj=True, max_iters=1)
    traj = r["traj"].cpu().numpy()
    prob.close()
    _, ref = oracle.bim_solve_batch([inst], np.zeros(n, np.int32), seqs, np.full(n, L, np.int32),
                                    opts=oracle.default_opts(max_iters=1), want_traj=True)
    for i in range(n):
        got = np.concatenate([traj[i][: 5 * (N + 1)], traj[i][5 * (N + 1): 17 * N + 5]]).astype(np.float64)
        scale = max(1.0, np.abs(ref[i]).max())
        assert np.max(np.abs(got - ref[i])) <= 1e-4 * max(1.0, N / 15) * scale, i
