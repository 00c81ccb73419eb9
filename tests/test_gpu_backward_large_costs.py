"""The replay's screen where its FP32 sums overflow though every value of the
solve is finite: a node's vector near 1.8e38 and tables near 1.7e38 (their sum
is beyond FP32; a = 1/2 (m1 + uh) and all that follows is not).  The gradient is
the all-FP64 replay's bit for bit."""
import numpy as np
import pytest

from paper_2004_08227_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pair(Lu, Lv, seed):
    rng = np.random.default_rng(seed)
    noise = lambda n: 1e35 * rng.random(n)
    unary = np.concatenate([0.8e38 + noise(Lu), 1.8e38 + noise(Lv)])
    table = 1.7e38 + noise(Lu * Lv)
    return W.Model(np.array([Lu, Lv], np.int32), np.zeros(1, np.int32), np.ones(1, np.int32),
                   unary.astype(np.float32), table.astype(np.float32))


@pytest.mark.parametrize("Lu,Lv", [(1, 1), (5, 7), (16, 16), (17, 30), (64, 33), (64, 64), (100, 128), (128, 97)])
def test_overflowing_screens(Lu, Lv):
    from paper_2004_08227_gb300.solver import Solver
    models = [_pair(Lu, Lv, 10 * Lu + Lv), W.complete(3, min(Lu, Lv), seed=1)]
    assert float(models[0].unary[Lu:].min()) + float(models[0].pairwise.min()) > float(np.finfo(np.float32).max)
    grads = []
    for fp64 in (False, True):
        with Solver(models, record_every=2, test_fp64_replay=fp64) as s:
            s.run(3)
            assert np.isfinite(s.bound()).all()
            grads.append(s.backward())
    np.testing.assert_array_equal(grads[0][0], grads[1][0])
    np.testing.assert_array_equal(grads[0][1], grads[1][1])
