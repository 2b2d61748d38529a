"""dem_contact_forces_noalloc over the sizes at which its warps change shape,
and a particle that many others come near without touching."""
import numpy as np
import pytest

from paper_2507_12610_gb300 import scenes
from tests.test_zz_no_alloc import TOL, env, noalloc, reference_first_step, rel  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 9, 33, 8191, 8192, 8193, 40960, 40961, 131072])
def test_every_warp_shape(env, n):  # noqa: F811
    torch, dem = env
    k = int(np.ceil(n ** (1.0 / 3.0)))
    s = scenes.lattice_box_scene((k, k, k), seed=n, spacing=1.95e-3, jitter=3e-5, speed=0.05,
                                 spin=30.0, walls=False)
    for key in ("R", "x", "v", "w", "q"):
        s[key] = np.ascontiguousarray(s[key][:n])
    rc, F, T = noalloc(torch, dem, s)
    assert rc == dem.DEM_OK
    F_ref, T_ref = reference_first_step(dem, s)
    if n == 1:
        assert not F.any() and not T.any()
        return
    assert np.abs(F_ref).max() > 0
    assert rel(F, F_ref) <= TOL and rel(T, T_ref) <= TOL


def test_many_near_and_few_touching(env):  # noqa: F811
    # 100 small spheres around a large one at a gap below the single-precision
    # margin of a half-metre box: none touches, and 100 is more than the
    # partners a particle may touch; then 60 of them pushed in
    torch, dem = env
    k = np.arange(100) + 0.5
    phi, th = np.arccos(1.0 - 2.0 * k / 100), np.pi * (1.0 + 5.0 ** 0.5) * k
    d = np.stack([np.cos(th) * np.sin(phi), np.sin(th) * np.sin(phi), np.cos(phi)], 1)
    R = np.concatenate([[1.0e-3], np.full(100, 5e-5), [1.0e-3]])
    gap = np.full(100, 1e-7)
    # cell edges (2 mm) through the large sphere's centre: few spheres a cell
    box = (np.full(3, -4e-3), np.array([0.504, 4e-3, 4e-3]))
    for pushed in (0, 60):
        gap[:pushed] = -1e-6
        x = np.vstack([[[0.0, 0.0, 0.0]], d * (R[0] + R[1] + gap)[:, None], [[0.5, 0.0, 0.0]]])
        s = dict(params=scenes.base_params(), R=R, x=x, v=np.zeros_like(x),
                 w=np.full_like(x, 3.0), q=None)
        rc, F, T = noalloc(torch, dem, s, box=box)
        assert rc == dem.DEM_OK
        touched = np.abs(F).max(axis=1) > 0
        assert touched[1:101].sum() == pushed and touched[0] == (pushed > 0)
    gap[:] = -1e-6
    s["x"][1:101] = d * (R[0] + R[1] + gap)[:, None]
    rc, _, _ = noalloc(torch, dem, s, box=box)
    assert rc == dem.DEM_ERR_CAPACITY
