"""Which driver the models of test_gpu_small_labels.py get: a driver that began to
refuse them would leave those tests without a comparison."""
import pytest

from test_gpu_small_labels import MODELS

pytestmark = pytest.mark.gpu

# more than 16 labels, or matchings of more edges than one step of a CTA takes
NARROW = ("ragged_31", "ragged_32", "full_32", "knn")
TOO_LARGE = ("knn",)  # for the resident driver: 367 KB of state


@pytest.mark.parametrize("name", list(MODELS))
def test_the_driver_that_runs(name):
    from paper_2004_08227_gb300._lib import MplppError
    from paper_2004_08227_gb300.solver import Solver
    models = MODELS[name]()
    with Solver(models) as s:
        inf = s.info()
        assert inf["mode"] == ("persistent" if name in NARROW else "resident")
        assert (inf["cluster"] == 0) == (name in NARROW)
    with Solver(models, mode="persistent") as s:
        assert s.info()["mode"] == "persistent" and s.info()["cluster"] == 0
    if name in TOO_LARGE:
        with pytest.raises(MplppError) as ei:
            Solver(models, mode="resident")
        assert ei.value.status == -7
    else:
        with Solver(models, mode="resident") as s:
            assert s.info()["mode"] == "resident" and s.info()["grid"] == len(models)
