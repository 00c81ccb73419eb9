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
    """K_n with integer costs (exact ties); its first edge leads to its last node,
    which alone has more than 300 labels."""
    m = W.uneven_complete(n, max(1, min(labels, 300) - 3), min(labels, 300), seed=seed)
    m.labels[-1] = labels
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


def _raises_timeout(call):
    with pytest.raises(MplppError) as ei:
        call()
    assert ei.value.status == TIMEOUT


@pytest.mark.parametrize("n,labels", [(2, 5), (30, 16), (20, 40), (12, 70), (4, 1025)])
def test_a_wait_of_the_rounding_runs_out(n, labels):
    """One team waits for a label that it never sees; the next call on the same
    solver, and another solver, work."""
    m = _tied(n, labels, n)
    with Solver([m], mode="looped", test_unreachable_wait=True, spin_limit=2000) as s, Solver([m], mode="looped") as good:
        s.run(1)
        _raises_timeout(s.labeling)
        good.run(1)
        assert np.array_equal(s.bound(), good.bound())
        x, _ = good.labeling()
        assert (x >= 0).all() and (x < m.labels).all()


@pytest.mark.parametrize("n,labels", [(6, 8), (6, 40), (5, 100), (3, 260)])
@pytest.mark.parametrize("fp64_replay", [False, True])
def test_a_wait_of_the_backward_runs_out(n, labels, fp64_replay):
    """The replay's queue (up to 128 labels), or with the all-FP64 replay, which
    waits for nothing, the sweep's."""
    m = W.complete(n, labels, seed=1)
    with Solver([m], mode="looped", record_every=2, test_unreachable_wait=True, spin_limit=2000,
                test_fp64_replay=fp64_replay) as s:
        s.run(3)
        _raises_timeout(s.backward)
        s.reset()
        s.run(1)
        s.sync()


@pytest.mark.parametrize("how", ["labeling", "backward"])
def test_a_low_limit_leaves_the_rounding_and_the_backward_alone(how):
    m = W.uneven_complete(40, 2, 30, seed=2)
    with Solver([m], mode="looped", record_every=2, spin_limit=1) as a, \
            Solver([m], mode="looped", record_every=2) as b:
        a.run(3)
        b.run(3)
        x, y = (a.labeling(), b.labeling()) if how == "labeling" else (a.backward(), b.backward())
        assert all(np.array_equal(p, q) for p, q in zip(x, y))


def _star(labels):
    rng = np.random.default_rng(7)
    labels = np.asarray(labels, np.int32)
    n = labels.shape[0]
    eu, ev = np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32)
    size = int((labels[eu].astype(np.int64) * labels[ev]).sum())
    return W.Model(labels, eu, ev, rng.random(int(labels.sum())).astype(np.float32),
                   rng.standard_normal(size).astype(np.float32))


@pytest.mark.parametrize("name,kw", [
    ("k10", {"cluster": 1, "threads": 128}),  # a CTA per edge, rows in registers
    ("k10", {"cluster": 2, "threads": 128}),  # a cluster per edge
    ("k10_40", {}),                           # the automatic mapping above 32 labels
    ("star_132", {"cluster": 1, "threads": 512}),             # wide rows, with a warp that polls
    ("k10", {}),                              # the narrow form
])
def test_a_wait_of_the_persistent_drivers_runs_out(name, kw):
    models = {"k10": lambda: W.complete(10, 8, seed=0), "k10_40": lambda: W.complete(10, 40, seed=0),
              "star_132": lambda: _star([40, 132, 132, 130, 131])}
    m = models[name]()
    with Solver([m], mode="persistent", test_unreachable_wait=True, spin_limit=2000, **kw) as s:
        assert s.info()["poller_warp"] == int(name == "star_132")
        s.run(3)
        _raises_timeout(s.sync)
    with Solver([m], mode="persistent", **kw) as s, Solver([m], mode="looped") as ref:
        s.run(3)
        ref.run(3)
        assert all(np.array_equal(x, y) for x, y in zip(s.state_arrays()[1:], ref.state_arrays()[1:]))
