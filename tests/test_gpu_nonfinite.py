"""Non-finite values stay with the Gaussians that meet them in the compositing adjoint: two
Gaussians in one warp's 8 x 4 sub-tile that share no pixel, the one behind with an infinite
feature, a NaN upstream gradient at one of its pixels, or an alpha of 1 (no transmittance left
behind it).  The gradients of the other one are bit for bit those of the finite scene: its sums
run over the same terms, in one warp."""
import numpy as np
import pytest
import torch

import synthetic
from helpers import FWD_ABS
from test_gpu_parity import f32_camera, make

pytestmark = pytest.mark.gpu

W, H = 16, 8
GEOMETRY = ("mean", "log_scale", "quat", "opacity_logit")
CFGS = [(4, dict(tile_w=16, tile_h=8)), (16, dict(tile_w=16, tile_h=8)), (40, dict(tile_w=8, tile_h=8)),
        (16, dict(tile_w=8, tile_h=8, half_masks=True)),
        (32, dict(tile_w=8, tile_h=8, half_masks=True, half_tile_fwd=True))]


def _scene(C, seed):
    """Gaussian 0 at (1, 1.5) and, behind it, Gaussian 1 at (6, 1): deviations of at most 0.45
    pixels, so that alpha reaches 1/255 within 2.3 pixels, and the two share none."""
    f, rng = 16.0, np.random.default_rng(seed)
    uv, z = np.array([[1.0, 1.5], [6.0, 1.0]]), np.array([1.0, 2.0])
    mean = np.stack([(uv[:, 0] - 7.0) / f * z, (uv[:, 1] - 3.0) / f * z, z], 1)
    a = lambda x: np.ascontiguousarray(x, dtype=np.float32)
    g = dict(mean=a(mean), log_scale=a(np.log(z[:, None] / f * [0.45, 0.3, 0.38])),
             quat=a([np.array([9.0, 1.0, 2.0, 3.0]) / 95 ** 0.5] * 2),
             opacity_logit=a([0.4, 0.4]), rgb=a(rng.uniform(0, 1, (2, 3))), sem=a(rng.normal(size=(2, C))))
    up = [a(rng.normal(size=n * W * H)) for n in (3, 1, C)]
    return g, f32_camera(synthetic.make_camera(W, H, f, f, 7.0, 3.0)), up


def _grads(g, cam, up, cfg):
    r, p = make(g, [cam], **cfg)
    r.forward(p)
    c = r.n_contrib.cpu().numpy().reshape(H, W)
    assert c.max() == 1 and c[:, :4].any() and c[1, 6] == 1 and not c[4:, :4].any()
    grads = {k: torch.zeros_like(v) for k, v in p.items()}
    r.backward(p, grads, dL=tuple(torch.tensor(u, device="cuda") for u in up))
    torch.cuda.synchronize()
    return {k: v[0].cpu() for k, v in grads.items()}


def _same(got, want, keys):
    for k in keys:
        assert bool(torch.isfinite(want[k]).all()) and float(want[k].abs().max()) > FWD_ABS, k
        assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("C, cfg", CFGS)
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_infinite_feature_behind(C, cfg, value):
    g, cam, up = _scene(C, C)
    want = _grads(g, cam, up, cfg)
    for k, i in (("sem", C - 1), ("rgb", 1)):
        bad = dict(g, **{k: g[k].copy()})
        bad[k][1, i] = value
        _same(_grads(bad, cam, up, cfg), want, (*GEOMETRY, "rgb", "sem"))


@pytest.mark.parametrize("C, cfg", CFGS)
@pytest.mark.parametrize("plane, keys", [(0, (*GEOMETRY, "sem")), (1, (*GEOMETRY[1:], "rgb", "sem")),
                                         (2, (*GEOMETRY, "rgb"))])
def test_nan_upstream_gradient_at_a_pixel(C, cfg, plane, keys):
    """Of the colour, the depth or the features.  (The gradient of that feature itself is a product
    over all pixels of the warp, w = 0 times NaN included, and the mean's takes in the depth's:
    those are NaN.)"""
    g, cam, up = _scene(C, C + 1)
    want = _grads(g, cam, up, cfg)
    up[plane][1 * W + 6] = np.nan
    _same(_grads(g, cam, up, cfg), want, keys)


@pytest.mark.parametrize("C, cfg", CFGS)
def test_opaque_pixel_behind(C, cfg):
    """alpha_max = 1 and T_min = 0: Gaussian 1 of opacity 1 leaves no transmittance at its mean."""
    g, cam, up = _scene(C, C + 2)
    cfg = dict(cfg, alpha_max=1.0, T_min=0.0)
    want = _grads(g, cam, up, cfg)
    bad = dict(g, opacity_logit=np.array([0.4, 40.0], np.float32))
    _same(_grads(bad, cam, up, cfg), want, (*GEOMETRY, "rgb", "sem"))
