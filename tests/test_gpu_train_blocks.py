"""REINFORCE step at the edges of the rollout's block shapes: one, two or four data points a block (the line lies at one
and two blocks for each of the 148 SMs), a last block that is not full, and records of the gradient sums in one and in
several lists of 256 points; fewest and most draft calls and scores.  Oracle and tolerances as in test_gpu_train.py: fp32
sums against fp64, 2e-5 of the largest gradient entry."""
import numpy as np
import pytest

import harness as H
from paper_2512_14069_b200 import workloads as W
from test_gpu_train import HP, Trainer, _compare, _theta

pytestmark = pytest.mark.gpu

CASES = [(1, 10, 8), (148, 1, 2), (149, 10, 8), (296, 32, 3), (297, 10, 16), (299, 4, 2), (2100, 2, 4)]


@pytest.fixture(scope="module")
def ctx():
    from paper_2512_14069_b200 import binding as rb
    c = rb.Context(0)
    yield c
    c.close()


def _problem(n, k, t_max):
    from oracle import train_oracle as T
    cfg = W.shrink(W.CONFIGS[2], cid=330, k=k, t_max=t_max)
    w = W.gate_weights(cfg)
    w["b2"][1] += np.float32(0.8)
    batch = W.train_batch(cfg, n, n)
    return w, batch, T.batch_loss_and_grad(w, *batch, t_max, **HP)


@pytest.mark.parametrize("n,k,t_max", CASES)
def test_train_block_shapes(ctx, n, k, t_max):
    w, batch, (loss, grad, infos) = _problem(n, k, t_max)
    tr = Trainer(ctx, n, k, t_max, _theta(w))
    dev = [H.to_dev(x) for x in batch]
    for _ in range(2):                                   # the second pass finds the first one's records in the workspace
        tr.step(*dev, step=0)
        _compare(tr, w, None, infos, loss, grad)
