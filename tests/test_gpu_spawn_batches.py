"""A spawn event tests several attempts at once: the spheres kept, and the draws
used, are those of taking the attempts one by one (the oracle), for numbers of
attempts around a batch, boxes that fill up, and boxes cut by a wall."""
import numpy as np
import pytest

from tests.test_gpu_spawn import dem, oracle_of, spawn_scene  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "mixed", "mixed64"])
@pytest.mark.parametrize("attempts", [1, 15, 16, 17, 33, 700])
def test_events_keep_the_oracle_s_spheres(dem, oracle_mod, attempts, precision):  # noqa: F811
    s = spawn_scene(n_max=300, attempts=attempts, every=2, seed=attempts)
    # the box reaches down to the resting spheres and the floor plate
    s["spawn"].update(lo=(-0.009, -0.009, 0.0008))
    sc = dem.Scene.from_dict(s, precision=precision)
    oc = oracle_of(oracle_mod, s)
    steps = 9 if attempts > 1 else 41
    sc.step(steps)
    oc.step(steps)
    assert sc.synchronize() == 0
    assert sc.active == oc.active > 42
    assert np.allclose(sc.radii(), oc.radii(), rtol=1e-14, atol=0)
    tol = 1e-12 if precision == 0 else 1e-5
    assert np.abs(sc.state()["x"] - oc.state()["x"]).max() <= tol * 0.9e-3
