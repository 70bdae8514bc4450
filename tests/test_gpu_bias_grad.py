"""Bias gradients of a training step: the same bits from the same batch,
however many splits it is summed in (one writer per split and bias, the splits
added in order), and the FP64 oracle's within the bound of test_gpu_mlp.py."""
import numpy as np
import pytest
import torch

import paper_2609_21803_gb300 as P
import workloads as W
from oracle import mlp as O

pytestmark = pytest.mark.gpu


# (intervals per segment, segments, width, bimanual, rows): 1 split, 3 ragged
# ones, 16 of the training batch, as many as the smallest network allows, and
# the largest number of biases
@pytest.mark.parametrize("K, L, width, bim, M", [(3, 2, 256, False, 255), (11, 5, 256, False, 801),
                                                 (20, 4, 256, False, 4096), (1, 1, 16, False, 20000),
                                                 (15, 11, 256, True, 1030)])
def test_bias_gradients(K, L, width, bim, M):
    inst = dict(W.bimanual_instance(1) if bim else W.push_l4_instance(1), knots_per_segment=K, max_segments=L)
    prob = P.Problem([inst])
    q = P.comet_proposal_create(prob.handle, dict(width=width, rows_cap=128))
    din, w, dout, n = P.comet_proposal_dims(q)
    rng = np.random.default_rng(M)
    dims = [din, w, w, w, dout]
    params = [(rng.uniform(-1, 1, (dims[l + 1], dims[l])) / np.sqrt(dims[l]), rng.uniform(-0.1, 0.1, dims[l + 1]))
              for l in range(4)]
    P.comet_proposal_set_params(q, O.flatten(params).astype(np.float32))
    X, T = rng.normal(size=(M, din)), rng.normal(size=(M, dout))
    Om = rng.uniform(0, 1, size=(M, dout)) * (rng.uniform(size=(M, dout)) < 0.5)
    x, t, om = (torch.from_numpy(a).cuda() for a in (O.bf16_bits(X).view(np.int16), T.astype(np.float32),
                                                     Om.astype(np.float32)))
    biases = []
    for _ in range(8):
        P.comet_proposal_train_batch(q, x, t, om, M, {"lr": 0.0})
        grad = np.zeros(n, np.float32)
        P.comet_proposal_get_params(q, None, grad)
        biases.append([b for _, b in O.unflatten(grad, din, w, dout)])
    Y, cache = O.forward(params, X, round_hidden=True)
    for l, (_, want) in enumerate(O.backward(params, cache, Y, T, Om, round_hidden=True)):
        assert np.linalg.norm(biases[0][l] - want) <= 1e-2 * np.linalg.norm(want), l
        for again in biases[1:]:
            assert np.array_equal(again[l].view(np.int32), biases[0][l].view(np.int32)), l
    P.comet_proposal_destroy(q)
    prob.close()
