"""The autotuner times a block shape only where it selects another kernel (no GPU: the
scenes are fakes that count)."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2507_12610_gb300 import batch, dem


class FakeScene:
    made = []

    @classmethod
    def from_dict(cls, b, **kw):
        cls.made.append((kw["skin"], kw["step_warps"]))
        return cls()

    def step(self, n):
        pass

    def synchronize(self):
        return 0

    def stats(self):
        return {"rebuilds": 0}

    def close(self):
        pass


@pytest.mark.parametrize("precision,rows,runs", [
    (dem.DEM_MIXED, 81920, 2), (dem.DEM_MIXED, 81921, 4), (dem.DEM_MIXED64, 40960, 2),
    (dem.DEM_MIXED64, 40961, 4), (dem.DEM_FP64, 500_000, 2)])
def test_one_run_where_the_block_shape_has_no_effect(precision, rows, runs):
    FakeScene.made = []
    best, table = batch.autotune({"R": np.ones(rows)}, precision=precision, skins=[0.1, 0.2],
                                 dem=SimpleNamespace(Scene=FakeScene))
    assert len(FakeScene.made) == runs
    assert [(r["skin"], r["step_warps"]) for r in table] == [(0.1, 4), (0.1, 8), (0.2, 4),
                                                             (0.2, 8)]
    assert best in table and (runs == 4 or best["step_warps"] == 4)
    if runs == 2:
        assert table[0]["ms_per_step"] == table[1]["ms_per_step"]
