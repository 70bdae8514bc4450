"""Which shape a launch of the pushing evaluator has: the one that was set, at
every size; the autotuner's pick; otherwise the default's rule.  Launches of
every shape that fill the SMs, cold and warm-started, give each order the
results that it has alone, bit for bit."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


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


def _problem(P, K, L):
    return P.Problem([dict(W.push_l4_instance(6), knots_per_segment=K, max_segments=L)])


def _orders(P, n, L, seed=8):
    seqs = np.random.default_rng(seed).integers(0, 12, (n, L)).astype(np.uint8)
    return torch.from_numpy(P.pack_mode_seqs(seqs).view(np.uint8).reshape(n, P.MODE_SEQ_BYTES)).cuda()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def test_a_set_shape_is_launched_at_every_size(P):
    prob = _problem(P, 20, 4)
    assert P.comet_debug_launch_shape(prob.handle, 10) == (1, False)  # the default's rule
    for w in (4, 3, 2, 1):
        P.comet_set_launch_config(prob.handle, w, 1)
        resident = _sms() * w
        for n in (1, 10, resident * 7 // 8, resident, resident * 5 // 4):
            assert P.comet_debug_launch_shape(prob.handle, n) == (w, False), n
        for n in (resident * 5 // 4 + 1, 10 * resident):
            assert P.comet_debug_launch_shape(prob.handle, n) == (w, w > 1), n
    prob.close()


def test_the_autotuner_keeps_what_it_timed(P):
    # N_max = 36 and 44: no other test tunes them
    prob = _problem(P, 12, 3)
    default = P.comet_get_launch_config(prob.handle)
    pick, times = P.comet_autotune(prob.handle, _orders(P, 40, 3), 40, 5)
    assert all(t > 0 for t in times)
    for n in (1, 40, 100000):  # as if set
        assert P.comet_debug_launch_shape(prob.handle, n)[0] == pick["warps_per_block"]
    later = _problem(P, 12, 3)  # not told by a sample that leaves SMs idle
    assert P.comet_get_launch_config(later.handle) == default
    later.close()
    prob.close()
    prob = _problem(P, 11, 4)
    n = _sms() * 16 * 2 + 1  # 16 warps are more than any candidate keeps on an SM
    pick, _ = P.comet_autotune(prob.handle, _orders(P, n, 4), n, 5)
    assert P.comet_debug_launch_shape(prob.handle, 10) == (1, False)
    w = pick["warps_per_block"]
    assert P.comet_debug_launch_shape(prob.handle, 100000) == (w, w > 1)
    later = _problem(P, 11, 4)
    assert P.comet_get_launch_config(later.handle) == pick
    later.close()
    prob.close()


@pytest.mark.parametrize("w", [1, 2, 3, 4])
@pytest.mark.parametrize("few", [False, True])
def test_full_launches_of_every_shape(P, w, few):
    K, L, m = 11, 3, 5
    prob = _problem(P, K, L)
    P.comet_set_launch_config(prob.handle, w, 1)
    b = 1 if few else P.comet_get_launch_config(prob.handle)["max_blocks_per_sm"]
    P.comet_set_launch_config(prob.handle, w, b)
    tiles = _sms() * b * w * 5 // 4 // m + 1
    n = tiles * m
    assert P.comet_debug_launch_shape(prob.handle, n) == (w, w > 1)
    d = _orders(P, m, L)
    alone = full = None
    for _ in range(2):  # cold, then warm-started from the iterates of the cold run
        a = prob.eval(d, warm=None if alone is None else alone["traj"], want_traj=True, max_iters=40)
        r = prob.eval(d.repeat(tiles, 1), warm=None if full is None else full["traj"], want_traj=True, max_iters=40)
        torch.cuda.synchronize()
        for k in a:
            x, y = a[k].cpu().numpy(), r[k].cpu().numpy()
            y = y.reshape((tiles,) + x.shape)
            assert (y.view(np.int32) == x.view(np.int32)[None]).all(), k
        alone, full = a, r
    prob.close()
