"""Spawning beside a thin triangle (16 mm by 10 um, in general position, every vertex first):
a sphere that overlaps it by a micrometre is refused, one a micrometre clear of it is kept,
as by the oracle.  Its closest point in single precision is off by up to 0.4 mm."""
import numpy as np
import pytest

from paper_2507_12610_gb300 import scenes
from tests.test_gpu_spawn import dem, oracle_of  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

R, LONG, THIN = 1.0e-3, 0.016, 1.0e-5


def needle(seed):
    """Vertices, unit vectors along and across the triangle, and its normal."""
    rng = np.random.default_rng(seed)
    e = rng.normal(size=3)
    e /= np.linalg.norm(e)
    n = np.cross(e, rng.normal(size=3))
    n /= np.linalg.norm(n)
    f = np.cross(n, e)
    return np.array([-0.5 * LONG * e, 0.5 * LONG * e, 0.43 * LONG * e + THIN * f]), e, f, n


@pytest.mark.parametrize("first", [0, 1, 2])
@pytest.mark.parametrize("precision", [0, 1, 2], ids=["fp64", "mixed", "mixed64"])
def test_spheres_at_a_needle_are_the_oracle_s(dem, oracle_mod, precision, first):  # noqa: F811
    kept = []
    for u in np.linspace(0.1, 0.85, 16):
        V, e, f, n = needle(int(1000 * u))
        for gap in (-1e-6, 1e-6):
            # above the inside of the face
            c = V[0] + u * LONG * e + 0.3 * u * THIN * f + (R + gap) * n
            s = dict(params=scenes.base_params(), R=np.zeros(0), x=np.zeros((0, 3)),
                     verts=np.roll(V, -first, axis=0), tris=np.array([[0, 1, 2]], np.int32),
                     tri_radius=None, spawn=dict(n_max=2, lo=c, hi=c, r_min=R, r_max=R,
                                                 attempts=3, seed=1))
            sc = dem.Scene.from_dict(s, precision=precision)
            oc = oracle_of(oracle_mod, s)
            sc.step(1)
            oc.step(1)
            assert sc.synchronize() == 0
            kept.append((sc.active, oc.active))
            assert oc.active == (1 if gap > 0 else 0)
            sc.close()
    wrong = sum(a != b for a, b in kept)
    assert wrong == 0, wrong
