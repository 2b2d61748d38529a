"""A grain at the hub of a drum's end cap is near all triangles of the fan: the scene states
that capacity, the list build holds them, and the contact is the oracle's."""
import math

import numpy as np
import pytest

from paper_2507_12610_gb300 import scenes


def distances(q, V, T):
    """From point q to every triangle of (V, T)."""
    A, B, C = V[T[:, 0]], V[T[:, 1]], V[T[:, 2]]
    n = np.cross(B - A, C - A)
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    h = np.einsum("ij,ij->i", q - A, n)
    foot = q - h[:, None] * n
    inside, best = np.ones(len(T), bool), np.full(len(T), np.inf)
    for P, E in ((A, B - A), (B, C - B), (C, A - C)):
        inside &= np.einsum("ij,ij->i", np.cross(E, foot - P), n) >= 0
        t = np.clip(np.einsum("ij,ij->i", q - P, E) / np.einsum("ij,ij->i", E, E), 0, 1)
        best = np.minimum(best, np.linalg.norm(q - P - t[:, None] * E, axis=1))
    return np.where(inside, np.abs(h), best)


@pytest.mark.parametrize("n,theta,rings,radius", [
    (1500, 32, 4, 0.022), (2000, 64, 8, scenes.drum_geometry(2000)[0] + 0.006),
    (20_000, 64, 8, None), (20_000, 128, 15, None)])
def test_the_scene_states_the_capacity_of_its_hub(n, theta, rings, radius):
    s = scenes.drum_scene(n=n, n_theta=theta, n_rings=rings, nn_dist=2.15e-3, radius=radius)
    R = 1.2e-3
    reach = 1.25 * R  # with the default skin
    x = -0.5 * s["drum_length"] + R
    r_in = s["drum_radius"] * math.cos(math.pi / theta) - R
    most = 0
    for rho in np.concatenate([[0.0], np.geomspace(1e-4, r_in, 40)]):
        for phi in (0.3, 0.3 + math.pi / theta):
            q = np.array([x, rho * math.cos(phi), rho * math.sin(phi)])
            most = max(most, int((distances(q, s["verts"], s["tris"]) < reach).sum()))
    assert most == theta > 16
    assert s["max_mesh_contacts"] >= most


def test_scenes_from_dicts_take_the_stated_capacity(monkeypatch):
    from paper_2507_12610_gb300 import dem
    seen = []
    monkeypatch.setattr(dem.Scene, "__init__", lambda self, *a, **k: seen.append(k))
    s = scenes.drum_scene(n=500, n_theta=64, n_rings=4, radius=0.02)
    dem.Scene.from_dict(s)
    dem.Scene.from_dict(s, max_mesh_contacts=3)
    dem.Scene.from_dict(scenes.box_scene(n=10))
    assert [k["max_mesh_contacts"] for k in seen] == [64, 3, 0]


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "mixed", "mixed64"])
def test_a_grain_at_the_hub_steps_as_the_oracle_s(oracle_mod, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_12610_gb300 import build, dem
    build.build()
    s = scenes.drum_scene(n=40, seed=3, n_theta=64, n_rings=4, radius=0.02, speed=0.0)
    # the first grain, pressed 2 um into the cap beside the hub
    s["x"][0] = (-0.5 * s["drum_length"] + s["R"][0] - 2e-6, 3e-4, 2e-4)
    sc = dem.Scene.from_dict(s, precision=precision, record_forces=True)
    V, El, rad = scenes.all_elements(s)
    oc = oracle_mod.OracleScene(s["params"], s["R"], s["x"], s["v"], s["w"], s["q"], V, El, rad)
    for steps in (1, 60):
        sc.step(steps)
        oc.step(steps)
        assert sc.synchronize() == 0
        F, Fo = sc.forces()[0], oc.forces()[0]
        tol = 1e-12 if precision == 0 else 1e-5
        assert steps > 1 or np.abs(Fo[0]).max() > 0  # (later it has come off the cap)
        assert np.abs(F - Fo).max() <= tol * np.abs(Fo).max()
        assert np.abs(sc.state()["x"] - oc.state()["x"]).max() <= tol * 0.8e-3
