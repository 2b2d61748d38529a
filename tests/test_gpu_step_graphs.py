"""Each step graph says for itself whether it loops on the device: a call takes all of its
steps also where one of the two graphs is a plain sequence (as the driver may leave it)."""
import numpy as np
import pytest

from tests.test_gpu_step_batches import dem, drum, run  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("plain", ["0", "8"], ids=["both_plain", "one_step_graph_plain"])
@pytest.mark.parametrize("precision", [0, 1])
def test_every_call_takes_its_steps(dem, monkeypatch, precision, plain):  # noqa: F811
    cuts = [2, 1, 3, 2, 8, 9, 16, 2, 17, 40]
    ref, stats = run(dem, drum(), precision, [sum(cuts)])
    monkeypatch.setenv("DEM_GRAPH_CONDITIONAL", plain)
    st, other = run(dem, drum(), precision, cuts)  # (run asserts the number of steps)
    assert other["rebuilds"] == stats["rebuilds"]
    for k in ref:
        assert np.array_equal(ref[k], st[k]), k
