"""Gradients against the FP64 oracle's reverse mode where the replay's and the
sweep's layouts turn: several warps per label vector, and beyond 256 labels
several labels per thread (up to the limit of 768)."""
import numpy as np
import pytest

import oracle
from oracle import schedule as osched
from paper_2004_08227_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-4  # relative, with a floor of 1e-3: gradients are sums of +-2^-k returned in FP32


def _close(g, ref):
    return np.abs(g - ref) <= TOL * np.maximum(np.abs(ref), 1e-3)


def _model(labels, seed):
    rng = np.random.default_rng(seed)
    labels = np.asarray(labels, np.int32)
    eu, ev = np.triu_indices(labels.shape[0], k=1)
    size = int((labels[eu].astype(np.int64) * labels[ev]).sum())
    return W.Model(labels, eu.astype(np.int32), ev.astype(np.int32), rng.random(int(labels.sum())).astype(np.float32),
                   rng.standard_normal(size).astype(np.float32), schedule="round_robin")


@pytest.mark.parametrize("labels", [(65, 64, 65, 63), (128, 127, 128), (129, 130, 128), (256, 255, 256), (257, 258, 256),
                                    (300, 290, 300), (512, 60, 90), (40, 513, 70), (70, 768, 50), (767, 30)])
@pytest.mark.parametrize("checkpoints", [False, True])
def test_wide_gradients_match_the_oracle(labels, checkpoints):
    from paper_2004_08227_gb300.solver import Solver
    T, weights = 4, [0.5, -2.0]
    models = [_model(labels, sum(labels)), _model(labels[:2], 1)]
    with Solver(models, record_every=3, test_checkpoints=checkpoints) as s:
        s.run(T)
        gu, gp = s.backward(weights)
    u = p = 0
    for m, w in zip(models, weights):
        order = osched.build(m.schedule, m.n, m.edge_u, m.edge_v)[1]
        _, ru, rp = oracle.grad(m, order, T)
        assert np.all(_close(gu[u:u + ru.size], w * ru)), np.abs(gu[u:u + ru.size] - w * ru).max()
        assert np.all(_close(gp[p:p + rp.size], w * rp)), np.abs(gp[p:p + rp.size] - w * rp).max()
        u, p = u + ru.size, p + rp.size
