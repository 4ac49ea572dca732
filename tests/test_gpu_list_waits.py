"""Failure detection of the list build's bounded waits, without a fault: one part of a step publishes
nothing, the waits for it run out after 1000 polls, the status says so, and the lists are empty:
nothing that the failed step left unwritten is used (the workspace and the lists hold poison).
The render of empty lists is the background, and the next build is right."""
import ctypes as C

import numpy as np
import pytest
import torch

import synthetic
from test_gpu_parity import f32_camera, make

pytestmark = pytest.mark.gpu

STEPS = dict(compaction=0, depth_first=1, depth_last=4, slots=5, culling=6, tile_first=7, tile_last=8, order=11)


def _build(r, step=None):
    from paper_2412_01217_gb300._lib import call
    from paper_2412_01217_gb300.splat import _ptr, _stream
    if step is None:
        return r.build_lists()
    call("sg_tile_lists_timeout_probe", C.byref(r._proj), r.N, r.V, _ptr(r.views), r.n_tiles, C.byref(r._ccfg),
         C.byref(r._lists), _ptr(r.tile_ws), r.tile_ws.numel(), step, 1000, _ptr(r.status), _stream())


def _state(r):
    torch.cuda.synchronize()
    K = r.instance_count()
    return int(r.status.item()), K, [t.clone() for t in (r.tile[:K], r.record[:K], r.ranges, r.order)]


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("step", STEPS)
def test_a_wait_that_runs_out_leaves_empty_lists(step, half):
    from paper_2412_01217_gb300._lib import STATUS_TIMEOUT
    g = synthetic.cloud_scene(30_000, 4, seed=5)
    cam = f32_camera(synthetic.make_camera(520, 400, 470.0, 470.0, 259.5, 199.5))
    r, p = make(g, [cam], tile_w=8, tile_h=8, half_masks=half, bg=(0.25, 0.5, 0.75))
    assert r.n_tiles == 65 * 50  # 12 bits: two tile passes; 13 parts of the work order
    r._lists.half_masks = int(half)
    r.project(p)
    _build(r)
    want = _state(r)
    assert want[0] == 0 and want[1] > 20_000  # every step has several parts
    for t in (r.tile_ws, r.tile, r.record, r.ranges, r.order):
        t.view(torch.uint8).fill_(0xff)
    _build(r, STEPS[step])
    status, K, (_, _, ranges, order) = _state(r)
    assert status == STATUS_TIMEOUT
    if step == "order":
        assert K == want[1] and all(torch.equal(a, b) for a, b in zip(_state(r)[2], want[2]))
    else:
        assert K == 0 and not ranges.any()
        assert torch.equal(order.cpu(), torch.arange(r.n_tiles, dtype=order.dtype))
        r.rasterize(p)
        torch.cuda.synchronize()
        assert bool((r.T_final == 1).all()) and not r.n_contrib.any()
        assert np.array_equal(r.img_rgb.view(3, -1)[:, 0].cpu().numpy(), np.float32([0.25, 0.5, 0.75]))
    r.status.zero_()
    _build(r)
    again = _state(r)
    assert again[:2] == want[:2] and all(torch.equal(a, b) for a, b in zip(again[2], want[2]))


def test_read_status_reports_the_timeout():
    from paper_2412_01217_gb300._lib import SgError
    g = synthetic.cloud_scene(30_000, 4, seed=5)
    r, p = make(g, [f32_camera(synthetic.make_camera(520, 400, 470.0, 470.0, 259.5, 199.5))], tile_w=8, tile_h=8)
    r.project(p)
    _build(r, STEPS["culling"])
    with pytest.raises(SgError) as e:
        r.check_status()
    assert e.value.code == 3 and "bounded device wait" in str(e.value)
