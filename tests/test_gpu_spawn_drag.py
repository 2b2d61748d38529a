"""A spawned grain feels the fluid's drag from its first step on: the same scenes as the
spawning tests with a viscosity, against the oracle at their bounds.  The grains start at
1 m/s, so a first step without drag moves one by c_i dt = 2e-5 of its speed, 1e4 times the
double-precision bound."""
import numpy as np
import pytest

from tests.test_gpu_spawn import dem, oracle_of, spawn_scene  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp64", "fp64_two_sided", "mixed", "mixed64"])
@pytest.mark.parametrize("steps", [1, 2, 31])
def test_first_step_of_a_spawned_grain_has_drag(dem, oracle_mod, monkeypatch, steps, mode):  # noqa: F811
    if mode == "fp64_two_sided":
        monkeypatch.setenv("DEM_FP64_TWO_SIDED", "1")
    s = spawn_scene(n_max=300)
    s["params"]["eta"] = 1.0e-3
    sc = dem.Scene.from_dict(s, precision={"mixed": 1, "mixed64": 2}.get(mode, 0))
    oc = oracle_of(oracle_mod, s)
    sc.step(steps)
    oc.step(steps)
    assert sc.synchronize() == 0
    assert sc.active == oc.active > 42
    a, b = sc.state(), oc.state()
    tol = 1e-12 if mode.startswith("fp64") else 1e-5
    assert np.abs(a["x"] - b["x"]).max() <= tol * 0.9e-3
    for k in ("v", "w"):
        assert np.abs(a[k] - b[k]).max() <= tol * np.abs(b[k]).max(), k
