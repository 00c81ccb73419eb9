"""The mapping that info() and the autotuner name can be asked for: a solver made
with that mode, cluster and threads is accepted, takes the same mapping and
computes the same state."""
import numpy as np
import pytest

from paper_2004_08227_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MODELS = {
    "tiny": lambda: [W.complete(5, 8, seed=1)],  # resident: a single warp
    "k20": lambda: [W.complete(20, 8, seed=2)],
    "labels_13": lambda: [W.complete(40, 13, seed=3)],
    "labels_32": lambda: [W.knn(200, 6, 32, seed=4)],
    "labels_40": lambda: [W.uneven_complete(9, 30, 40, seed=5)],
    "labels_140": lambda: [W.complete(5, 140, seed=6)],
}


def _again(models, mode, cluster, threads, T):
    from paper_2004_08227_gb300.solver import Solver
    with Solver(models, mode=mode, cluster=cluster, threads=threads) as s:
        s.run(T)
        return s.state_arrays(), s.info()


@pytest.mark.parametrize("mode", ["auto", "persistent", "resident"])
@pytest.mark.parametrize("name", list(MODELS))
def test_the_mapping_of_info_can_be_requested(name, mode):
    from paper_2004_08227_gb300.solver import Solver
    models = MODELS[name]()
    if mode == "resident" and name in ("labels_32", "labels_40", "labels_140"):
        pytest.skip("more labels or a larger state than the resident driver takes")
    with Solver(models, mode=mode) as s:
        inf = s.info()
        s.run(3)
        want = s.state_arrays()
    got, inf2 = _again(models, inf["mode"], inf["cluster"], inf["threads"], 3)
    assert np.array_equal(want[1], got[1]) and np.array_equal(want[2], got[2])
    assert [inf2[k] for k in ("mode", "cluster", "threads", "grid")] == \
        [inf[k] for k in ("mode", "cluster", "threads", "grid")]


@pytest.mark.parametrize("name", ["tiny", "k20", "labels_32"])
def test_the_mappings_of_the_autotuner_can_be_requested(name):
    from paper_2004_08227_gb300.solver import Solver
    models = MODELS[name]()
    with Solver(models) as s:
        rep = s.autotune(1)
        inf = s.info()
        s.run(2)
        want = s.state_arrays()
    best = rep["best"]
    assert [inf["mode"], inf["cluster"], inf["threads"]] == [best["mode"], best["cluster"], best["threads"]]
    for cluster, threads, mode, _ in rep["candidates"]:
        got, _ = _again(models, mode, cluster, threads, 2)
        assert np.array_equal(want[1], got[1]) and np.array_equal(want[2], got[2]), (mode, cluster, threads)
