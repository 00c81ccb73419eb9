"""Waits on the device that run out: the call ends with MPLPP_E_TIMEOUT, reads
nothing outside its arrays on the way, and the device stays usable."""
import numpy as np
import pytest

from paper_2004_08227_gb300 import workloads as W
from paper_2004_08227_gb300._lib import MplppError
from paper_2004_08227_gb300.solver import Solver

pytestmark = pytest.mark.gpu

TIMEOUT = -4


def _tied(n, labels, seed):
    """K_n with integer costs (exact ties); its first edge leads to its last node."""
    m = W.uneven_complete(n, max(1, labels - 3), labels, seed=seed)
    k = np.random.default_rng(seed).permutation(m.E)
    k = np.concatenate([[m.E - 1], k[k != m.E - 1]])
    size = int((m.labels[m.edge_u].astype(np.int64) * m.labels[m.edge_v]).sum())
    rng = np.random.default_rng(seed + 1)
    return W.Model(m.labels, m.edge_u[k], m.edge_v[k], rng.integers(0, 3, int(m.labels.sum())).astype(np.float32),
                   rng.integers(0, 3, size).astype(np.float32))


@pytest.mark.parametrize("n,labels", [(200, 9), (120, 40), (60, 70)])
def test_rounding_after_a_timed_out_run_without_sync(n, labels):
    """The rounding finds the run's timeout in the error word and stops waiting
    for neighbours that have no label yet; tied labels are then summed again."""
    m = _tied(n, labels, n)
    with Solver([m], mode="queue", test_unreachable_wait=True, spin_limit=2000) as s:
        s.run(2)
        with pytest.raises(MplppError) as ei:
            s.labeling()
        assert ei.value.status == TIMEOUT
        with Solver([m]) as good:
            good.run(2)
            x, _ = good.labeling()
            assert (x >= 0).all() and (x < m.labels).all()


def test_a_low_limit_leaves_the_automatic_structured_driver_alone():
    """spin_limit = 1 ends waits of the drivers that a caller asked for; AUTO's
    structured driver took a launch per matching, without waits, before it ran
    from the queue."""
    m = W.grid_trunc_linear(12, 13, 20, weight=1.0, tau=4.0, seed=1)
    with Solver([m], spin_limit=1) as a, Solver([m], mode="looped") as b:
        assert a.info()["mode"] == "structured" and a.info()["launches_per_iteration"] == 0
        a.run(20)
        b.run(20)
        a.sync()
        assert all(np.array_equal(x, y) for x, y in zip(a.state_arrays()[1:], b.state_arrays()[1:]))
