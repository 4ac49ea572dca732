"""Loss terms whose partial sums leave the range of a float: the means are finite and are returned
(the sums over a view run in double there), and infinite or NaN pixels make their own term so."""
import numpy as np
import pytest
import torch

import synthetic
from test_gpu_parity import f32_camera

pytestmark = pytest.mark.gpu

W, H, C = 256, 96, 8


def _terms(mode, depth=None, sem=None, levels=1):
    from paper_2412_01217_gb300 import LossConfig, PyramidRasterizer
    cam = f32_camera(synthetic.make_camera(W, H, float(W), float(W), W / 2 - 0.5, H / 2 - 0.5))
    r = PyramidRasterizer(1, C, [cam], levels, loss_cfg=LossConfig(sem_mode=mode, n_classes=C, check_numeric=True))
    P = r.P
    one = lambda n: torch.full((n * P,), 0.5, device="cuda")
    gt = dict(rgb=one(3), depth=one(1), sem=one(C), label=torch.zeros(P, dtype=torch.int32, device="cuda"))
    r.loss(gt, rendered=(one(3), one(1) if depth is None else depth(P), one(C) if sem is None else sem(P)))
    torch.cuda.synchronize()
    return r.terms.view(-1, 4)[0].tolist(), int(r.status.item())


@pytest.mark.parametrize("mode", ["ce", "paper"])
@pytest.mark.parametrize("d", [1e30, 1e36])
def test_depth_sum_beyond_float(mode, d):
    """24576 pixels that are each 1e36 off: their sum is 2.5e40, that of 256 of them 2.6e38."""
    (L_r, L_d, L_s, total), status = _terms(mode, depth=lambda P: torch.full((P,), d, device="cuda"))
    assert L_d == pytest.approx(d, rel=1e-5) and total == pytest.approx(d, rel=1e-5)
    assert np.isfinite([L_r, L_s]).all() and status == 0


def test_cross_entropy_sum_beyond_float():
    def sem(P):  # the labelled class 1e36 below the others: CE = 1e36 + ln 7
        s = torch.zeros(C, P, device="cuda")
        s[0] = -1e36
        return s.reshape(-1)
    (_, _, L_s, total), status = _terms("ce", sem=sem)
    assert L_s == pytest.approx(1e36, rel=1e-5) and total == pytest.approx(1e36, rel=1e-5) and status == 0


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_a_pixel_that_is_not_finite(value):
    from paper_2412_01217_gb300._lib import STATUS_NUMERIC

    def depth(P):
        t = torch.full((P,), 0.75, device="cuda")
        t[P // 2] = value
        return t
    (L_r, L_d, L_s, total), status = _terms("ce", depth=depth)
    assert np.isfinite([L_r, L_s]).all() and status == STATUS_NUMERIC
    assert np.array_equal([L_d, total], [value, value], equal_nan=True)
