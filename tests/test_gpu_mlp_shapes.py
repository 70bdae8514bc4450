"""The proposal's network over its whole range of layouts, against the FP64
oracle with the bounds of test_gpu_mlp.py: the fused forward at every input
width, one to several output blocks (split over CTAs when the tiles are few,
ragged last blocks and rows), widths that the layered GEMMs take, and a
training step with every kind of ragged tile, from device arrays with and
without 16-byte alignment."""
import numpy as np
import pytest
import torch

import paper_2609_21803_gb300 as P
import workloads as W
from oracle import mlp as O

pytestmark = pytest.mark.gpu


def _proposal(K, L, width, bim=False):
    d = dict(W.bimanual_instance(1) if bim else W.push_l4_instance(1), knots_per_segment=K, max_segments=L)
    prob = P.Problem([d])
    q = P.comet_proposal_create(prob.handle, dict(width=width, rows_cap=128))
    din, w, dout, n = P.comet_proposal_dims(q)
    rng = np.random.default_rng(K * 100 + L)
    d = [din, w, w, w, dout]
    params = [(rng.uniform(-1, 1, (d[l + 1], d[l])) / np.sqrt(d[l]), rng.uniform(-0.1, 0.1, d[l + 1]))
              for l in range(4)]
    P.comet_proposal_set_params(q, O.flatten(params).astype(np.float32))
    return prob, q, params, d


# (intervals per segment, segments, width, bimanual): in_dim, out_dim
SHAPES = [(3, 2, 256, False),    # 64, 32
          (11, 5, 256, False),   # 128, 176
          (7, 9, 256, False),    # 192, 192
          (11, 16, 256, False),  # 256, 544: blocks of 256, 256, 32
          (4, 2, 256, True),     # 128, 112
          (15, 6, 256, True),    # 192, 1088: five blocks
          (9, 4, 48, False),     # 64, 112 on the layered GEMMs
          (15, 11, 256, True)]   # 384, 1984: past the fused input width


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("M", [1, 129, 1300])
def test_forward(shape, M):
    prob, q, params, d = _proposal(*shape)
    X = np.random.default_rng(M).normal(size=(M, d[0]))
    y = np.zeros((M, d[-1]), np.float32)
    P.comet_proposal_forward(q, O.bf16_bits(X), M, y)
    want, _ = O.forward(params, X, round_hidden=True)
    rms = np.sqrt(np.mean(want ** 2))
    assert np.max(np.abs(y - want) / (np.abs(want) + rms)) <= 1e-2
    P.comet_proposal_destroy(q)
    prob.close()


@pytest.mark.parametrize("shape", [SHAPES[0], SHAPES[3], SHAPES[5], SHAPES[6]])
@pytest.mark.parametrize("M, offset", [(63, 0), (300, 1), (1025, 0)])
def test_training_step(shape, M, offset):
    prob, q, params, d = _proposal(*shape)
    rng = np.random.default_rng(M)
    X, T = rng.normal(size=(M, d[0])), rng.normal(size=(M, d[-1]))
    Om = rng.uniform(0, 1, size=(M, d[-1])) * (rng.uniform(size=(M, d[-1])) < 0.5)

    def dev(a):  # `offset` elements past an aligned address
        t = torch.zeros(a.size + offset, dtype=torch.from_numpy(a).dtype, device="cuda")
        t[offset:] = torch.from_numpy(a.reshape(-1)).cuda()
        return t[offset:]

    x = dev(O.bf16_bits(X).view(np.int16))
    loss = P.comet_proposal_train_batch(q, x, dev(T.astype(np.float32)), dev(Om.astype(np.float32)), M, {"lr": 0.0})
    n = sum(w.size + b.size for w, b in params)
    grad = np.zeros(n, np.float32)
    P.comet_proposal_get_params(q, None, grad)
    Y, cache = O.forward(params, X, round_hidden=True)
    assert loss == pytest.approx(O.loss(Y, T, Om), rel=1e-2)
    want = O.backward(params, cache, Y, T, Om, round_hidden=True)
    got = O.unflatten(grad.astype(np.float64), d[0], d[1], d[-1])
    for l in range(4):
        for a, b in zip(got[l], want[l]):
            assert np.linalg.norm(a - b) <= 1e-2 * np.linalg.norm(b), l
    P.comet_proposal_destroy(q)
    prob.close()
