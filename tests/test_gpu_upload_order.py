"""Scenes created and loaded while other streams keep the copy engines busy: the kernels that
follow an upload (element cell lists, poses, the first list build) read what was uploaded."""
import numpy as np
import pytest

from paper_2507_12610_gb300 import scenes
from tests.test_gpu_spawn import dem  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def test_kernels_after_an_upload_read_it(dem):  # noqa: F811
    import torch
    s = scenes.lattice_box_scene((5, 5, 5), seed=2, spacing=1.9e-3, jitter=2e-5, speed=0.05,
                                 mesh_omega=(0.0, 0.0, 3.0))
    ref = dem.Scene.from_dict(s, precision=1)
    ref.step(40)
    want, stats = ref.state(), ref.stats()
    assert stats["mesh_contacts"] > 0
    host = torch.empty(1 << 24, dtype=torch.uint8).pin_memory()
    there = [torch.empty(1 << 24, dtype=torch.uint8, device="cuda") for _ in range(3)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    for k in range(60):
        for st, buf in zip(streams, there):
            with torch.cuda.stream(st):
                buf.copy_(host, non_blocking=True)
        sc = dem.Scene.from_dict(s, precision=1, stream=streams[k % 3].cuda_stream if k % 2 else None)
        blob = sc.save()
        sc.step(40)
        assert sc.synchronize() == 0
        got = [(sc.state(), sc.stats())]
        sc.load(blob)
        sc.step(40)
        assert sc.synchronize() == 0
        got.append((sc.state(), sc.stats()))
        for st, other in got:
            assert other["mesh_contacts"] == stats["mesh_contacts"]
            for key in want:
                assert np.array_equal(st[key], want[key]), (k, key)
        sc.close()
