"""Steps run in batches on the device (a loop node of a CUDA graph): however a
run is cut into dem_step calls, and with the plain graphs (no conditional
nodes) too, the result is bitwise the same."""
import numpy as np
import pytest

from paper_2507_12610_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dem():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_12610_gb300 import build
    build.build()
    from paper_2507_12610_gb300 import dem as d
    d.load()
    return d


def drum():
    return scenes.drum_scene(n=1500, seed=4, n_theta=32, n_rings=4, nn_dist=2.15e-3, radius=0.022,
                             speed=0.5)


def heap():
    return scenes.repose_scene(n=300, seed=3, every=3)


def run(dem, s, precision, cuts):
    sc = dem.Scene.from_dict(s, precision=precision)
    for k in cuts:
        sc.step(k)
    assert sc.synchronize() == 0
    st, stats = sc.state(), sc.stats()
    sc.close()
    assert stats["steps"] == sum(cuts)
    return st, stats


@pytest.mark.parametrize("scene", [drum, heap], ids=["drum", "heap"])
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "mixed", "mixed64"])
def test_same_bits_however_the_steps_are_cut(dem, monkeypatch, scene, precision):
    s = scene()
    ref, stats = run(dem, s, precision, [200])
    assert stats["rebuilds"] > 2  # a rebuild inside a batch
    for cuts in ([1] * 17 + [2, 3, 7, 8, 9, 16, 17, 121], [199, 1]):
        st, other = run(dem, s, precision, cuts)
        assert other["rebuilds"] == stats["rebuilds"]
        for k in ref:
            assert np.array_equal(ref[k], st[k]), (cuts[:3], k)
    monkeypatch.setenv("DEM_GRAPH_CONDITIONAL", "0")
    st, _ = run(dem, s, precision, [200])
    for k in ref:
        assert np.array_equal(ref[k], st[k]), k


@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "mixed", "mixed64"])
@pytest.mark.parametrize("n", [1, 7, 9, 777])
def test_same_bits_for_any_number_of_rows(dem, precision, n):
    # the step kernels give a warp 8, 16 or 32 particles by the number of rows
    # of the scene; rows that await spawning (none is spawned here) change that
    # number and nothing else
    s = scenes.drum_scene(n=n, seed=6, n_theta=32, n_rings=4, nn_dist=2.0e-3, radius=0.018,
                          speed=0.5)
    ref, stats = run(dem, s, precision, [60])
    for rows in (8193, 32769, 40961, 81921):
        s["spawn"] = dict(n_max=rows, lo=(0, 0, 0), hi=(0, 0, 0), r_min=1e-3, r_max=1e-3,
                          attempts=0)
        st, other = run(dem, s, precision, [60])
        assert other["pair_contacts"] == stats["pair_contacts"]
        assert other["mesh_contacts"] == stats["mesh_contacts"]
        for k in ref:
            assert np.array_equal(ref[k], st[k][:n]), (rows, k)
