"""The loss kernels at the edges of their work split: images smaller than, equal to and just past
the 32 x 32 loss tiles (single rows and columns among them), semantic planes dealt to one, two and
three groups' CTAs, and a view whose partial sums take several rounds of the finalising
cluster.  Every term and gradient against the oracle, with the parity tolerances."""
import numpy as np
import pytest
import torch

import oracle
from helpers import check_close
from test_gpu_parity import f32_camera

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode, C", [("paper", 4), ("paper", 8), ("ce", 8)])
@pytest.mark.parametrize("W, H, levels", [(1, 1, 1), (5, 70, 1), (70, 5, 2), (31, 33, 1), (32, 32, 2), (33, 65, 3),
                                          (43, 22, 1), (700, 500, 1)])
def test_loss_at_tile_edges_matches_oracle(W, H, levels, mode, C):
    import synthetic
    from paper_2412_01217_gb300 import LossConfig, PyramidRasterizer
    rng = np.random.default_rng(W + 1000 * H + C)
    cam = f32_camera(synthetic.make_camera(W, H, float(W), float(W), W / 2 - 0.5, H / 2 - 0.5))
    r = PyramidRasterizer(1, C, [cam], levels, loss_cfg=LossConfig(sem_mode=mode, n_classes=C))
    P = r.P
    f = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    rend = (f(rng.uniform(size=3 * P)), f(rng.uniform(1, 3, size=P)), f(rng.normal(size=C * P)))
    gt = dict(rgb=f(rng.uniform(size=3 * P)), depth=f(rng.uniform(1, 3, size=P)),
              label=torch.tensor(rng.integers(0, C, size=P), dtype=torch.int32, device="cuda"),
              sem=f(rng.uniform(size=C * P)))
    r.loss(gt, rendered=rend)
    terms = r.terms.view(-1, 4).cpu().numpy()
    for v in range(r.V):
        sl = lambda t, n: r.view_slice(t, v, n).cpu().numpy().astype(np.float64)
        sem = sl(gt["sem"], C) if mode == "paper" else r.view_slice(gt["label"], v, 1)[0].cpu().numpy()
        tot, tm, gr = oracle.level_loss(sl(rend[0], 3), sl(rend[1], 1)[0], sl(rend[2], C), sl(gt["rgb"], 3),
                                        sl(gt["depth"], 1)[0], sem, sem_mode=mode)
        for got, want in zip(terms[v], (tm["L_r"], tm["L_d"], tm["L_s"], tot)):
            assert got == pytest.approx(want, rel=1e-5)
        for name, buf, n in (("rgb", r.dL_rgb, 3), ("depth", r.dL_depth, 1), ("sem", r.dL_sem, C)):
            got = r.view_slice(buf, v, n).cpu().numpy()
            ref = gr[name].reshape(got.shape)
            check_close(f"dL/d{name} v{v}", got, ref, 1e-4, 1e-4 * np.abs(ref).max())
