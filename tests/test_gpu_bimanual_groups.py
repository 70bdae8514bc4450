"""First iterate of the bimanual evaluator at horizons around its strides and
copy rings, against the FP64 oracle, each group of the record on a scale of its
own: poses, hand offsets, kinematic controls, forces in units of m g.

The bounds are four times the largest error that the kernel of another layout
(a lane per constraint row, one stage at a time) had over 13 horizons of 1..180
stages, three instances and 32 orders each: 7.9e-6, 0, 1.1e-5 and 5.4e-5, with
no growth along the horizon that a bound would have to follow."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

KINEMATIC = [0, 1, 2, 5, 8, 11]  # box rates, sliding rates, pressure centre
FORCES = [3, 4, 6, 7, 9, 10]     # both hands and the ground


@pytest.mark.parametrize("K, L", [(1, 1), (2, 1), (3, 1), (4, 1), (5, 1), (8, 1), (9, 1), (12, 1), (13, 1), (17, 2),
                                  (64, 2), (43, 3), (60, 3)])
def test_first_iterate_by_groups(K, L):
    import paper_2609_21803_gb300 as P
    N, n = K * L, 32
    inst = dict(W.bimanual_instance(8), knots_per_segment=K, max_segments=L)
    rng = np.random.default_rng(200 + N)
    seqs = [tuple(int(m) for m in rng.integers(0, 507, L)) for _ in range(n)]
    prob = P.Problem([inst])
    d = torch.from_numpy(P.pack_mode_seqs(seqs).view(np.uint8).reshape(n, P.MODE_SEQ_BYTES)).cuda()
    got = prob.eval(d, want_traj=True, max_iters=1)["traj"].cpu().numpy().astype(np.float64)
    prob.close()
    _, ref = oracle.bim_solve_batch([inst], np.zeros(n, np.int32), seqs, np.full(n, L, np.int32),
                                    opts=oracle.default_opts(max_iters=1), want_traj=True)
    mg = inst["mass"] * 9.81
    for i in range(n):
        x, xr = (a[: 5 * (N + 1)].reshape(5, N + 1) for a in (got[i], ref[i]))
        u, ur = (a[5 * (N + 1): 17 * N + 5].reshape(12, N) for a in (got[i], ref[i]))
        for name, a, b, unit, bound in (("poses", x[:3], xr[:3], 1.0, 3.2e-5), ("offsets", x[3:], xr[3:], 0.1, 1e-6),
                                        ("kinematic", u[KINEMATIC], ur[KINEMATIC], 1.0, 4.4e-5),
                                        ("forces", u[FORCES], ur[FORCES], mg, 2.2e-4)):
            assert np.abs(a - b).max() <= bound * max(unit, np.abs(b).max()), (name, i)
