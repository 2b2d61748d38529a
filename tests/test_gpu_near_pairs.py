"""The overlap pre-test of DEM_FP64 and DEM_MIXED64 works on chopped coordinates:
whatever the distance from the origin it lets every touching pair through, and the
law's exact test keeps the others out."""
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


def pairs(offset):
    """64 pairs on a lattice, overlapping or apart by parts of R_i + R_j from 1e-3 down
    to 1e-9 (1e-8 at the far offsets, where a coordinate's last bit is 1e-10 of it)."""
    s = scenes.box_scene(n=128, seed=6, gravity=False, size=(0.08, 0.08, 0.08))
    rng = np.random.default_rng(7)
    part = np.resize([1e-3, 1e-4, 1e-6, 1e-8, 1e-9 if abs(offset) < 10 else 1e-8], 64)
    part *= rng.choice([-1.0, 1.0], 64)
    n = rng.normal(size=(64, 3))
    n /= np.linalg.norm(n, axis=1)[:, None]
    k = np.arange(64)
    c = np.stack([k % 4, k // 4 % 4, k // 16], axis=1) * 0.016 + np.array([-0.024, -0.024, 0.016])
    d = (s["R"][0::2] + s["R"][1::2]) * (1.0 - part)
    x = np.empty((128, 3))
    x[0::2], x[1::2] = c + 0.5 * d[:, None] * n, c - 0.5 * d[:, None] * n
    lo, hi = s["domain"]
    s.update(x=x + offset, verts=s["verts"] + offset, domain=(lo + offset, hi + offset))
    d2 = np.linalg.norm(s["x"][0::2] - s["x"][1::2], axis=1)
    return s, int(np.sum(s["R"][0::2] + s["R"][1::2] >= d2))


@pytest.mark.parametrize("offset", [0.0, 1.0, -37.0, 1000.0])
@pytest.mark.parametrize("precision", [0, 2], ids=["fp64", "mixed64"])
def test_touching_pairs_are_found_far_from_the_origin(dem, offset, precision):
    s, touching = pairs(offset)
    assert 16 < touching < 48
    sc = dem.Scene.from_dict(s, precision=precision)
    sc.step(1)
    assert sc.synchronize() == 0
    got = sc.stats()["pair_contacts"]
    sc.close()
    assert got == touching
