"""The projection writes every record: a culled one has an empty rectangle and zero geometry and
extents, whatever the buffers held before (the poses of a rasterizer change between calls)."""
import pytest
import torch

import synthetic
from test_gpu_parity import f32_camera, make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iso", [False, True])
def test_culled_records_are_zero(iso):
    g = synthetic.cloud_scene(3000, 4, seed=8)
    g["mean"][::3, 2] *= -1  # behind the camera
    cams = [f32_camera(synthetic.make_camera(160, 120, 150.0, 150.0, cx, 59.5)) for cx in (79.5, 700.0)]
    r, p = make(g, cams, levels=2, isotropic=iso)
    for t in (r.geo, r.rect, r.ext):
        t.view(torch.uint8).fill_(0xff)
    r.project(p)
    torch.cuda.synchronize()
    rect = r.rect.view(-1, 2)
    culled = rect[:, 0] == rect[:, 1]
    assert 2000 < int(culled.sum()) < len(rect) - 500
    assert bool((rect[culled] == 0).all())
    assert bool((r.geo.view(-1, 8)[culled] == 0).all()) and bool((r.ext.view(-1, 2)[culled] == 0).all())
    assert bool(torch.isfinite(r.ext.view(-1, 2)).all())
