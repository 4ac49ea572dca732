"""Edges of the list build's radix passes and of the compositing kernels' 16-entry chunks.

* Lists of every digit width of the tile sort's last pass (one tile to 825 tiles), with enough
  instances for many parts of the chained scan, built repeatedly: always the same lists, in
  (tile, depth bits, record) order, with the ranges and the work order they imply.
* One small image behind stacks of 1 to 65 Gaussians (chunks of 16 with every kind of
  remainder): every pixel and all gradients against the oracle, with the parity tolerances.
"""
import numpy as np
import pytest
import torch

import oracle
import synthetic
from helpers import AMBIGUOUS_GRAD, FWD_ABS, FWD_REL, check_close, check_grads, ref_render
from test_gpu_parity import KEYS, _check_ranges_and_order, _gpu_lists, f32_camera, make, view_images

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W, H, levels, tile, half", [
    (16, 16, 1, (16, 16), False),    # 1 tile: one 1-bit pass
    (64, 48, 1, (16, 16), False),    # 12 tiles: 4 bits
    (160, 120, 1, (16, 16), False),  # 80 tiles: 7 bits
    (320, 180, 3, (16, 16), False),  # 315 tiles: passes of 5 and 4 bits
    (256, 128, 1, (8, 8), True),     # 512 tiles: 5 and 4 bits, half masks
    (520, 400, 1, (16, 16), False),  # 825 tiles: 5 and 5 bits
])
def test_lists_are_sorted_and_repeatable_for_every_digit_width(W, H, levels, tile, half):
    N = 20_000
    g = synthetic.cloud_scene(N, 4, seed=W + H)
    cam = f32_camera(synthetic.make_camera(W, H, 0.9 * W, 0.9 * W, W / 2 - 0.5, H / 2 - 0.5))
    r, p = make(g, [cam], levels=levels, tile_w=tile[0], tile_h=tile[1], half_masks=half)
    r.project(p)
    first = None
    for _ in range(25):
        r.build_lists()
        K, tiles, recs, ranges = _gpu_lists(r)
        if first is None:
            first = (tiles, recs)
            _check_ranges_and_order(r, tiles, ranges)
            depth = r.geo.view(-1, 8)[:, 2].contiguous().view(torch.int32).cpu().numpy()[recs]
            assert np.array_equal(np.lexsort((recs, depth, tiles)), np.arange(K))
            assert K >= 10_000 and len(np.unique(np.stack([tiles, recs]), axis=1)[0]) == K
            local = recs // N  # the tile's view is the record's
            off = np.array([v.tile_offset for v in r.views_host])
            assert np.array_equal(np.searchsorted(off, tiles, "right") - 1, local)
        assert np.array_equal(tiles, first[0]) and np.array_equal(recs, first[1])


def _stack(n, C, seed):
    """n Gaussians in front of a 16 x 8 camera, each reaching much of the image, faint enough
    that all of them contribute."""
    rng = np.random.default_rng(seed)
    z = rng.uniform(1.0, 3.0, n)
    mean = np.stack([rng.uniform(-0.35, 0.35, n) * z, rng.uniform(-0.15, 0.15, n) * z, z], 1)
    q = rng.normal(size=(n, 4))
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    return dict(mean=f(mean), log_scale=f(rng.uniform(np.log(0.1), np.log(0.5), (n, 3))),
                quat=f(q / np.linalg.norm(q, axis=1, keepdims=True)), opacity_logit=f(rng.normal(-2.5, 0.5, n)),
                rgb=f(rng.uniform(0, 1, (n, 3))), sem=f(rng.normal(size=(n, C))))


@pytest.mark.parametrize("C, cfg", [
    (4, dict(tile_w=16, tile_h=8, pixels_per_thread=1, pixels_per_thread_bwd=1)),
    (8, dict(tile_w=8, tile_h=8, pixels_per_thread=2, pixels_per_thread_bwd=2, batch=16)),
    (16, dict(tile_w=16, tile_h=16, pixels_per_thread=4, pixels_per_thread_bwd=4, batch=32)),
    (32, dict(tile_w=8, tile_h=8, pixels_per_thread=1, pixels_per_thread_bwd=1, half_masks=True)),
    (40, dict(tile_w=8, tile_h=8, pixels_per_thread=1, pixels_per_thread_bwd=1, half_masks=True, half_tile_fwd=True)),
])
@pytest.mark.parametrize("n", [1, 4, 15, 16, 17, 31, 33, 48, 65])
def test_stacks_around_the_chunk_size_match_oracle(n, C, cfg):
    W, H = 15, 7  # ragged in every tile shape
    g = _stack(n, C, seed=100 * n + C)
    cam = f32_camera(synthetic.make_camera(W, H, 16.0, 16.0, 7.0, 3.0))
    r, p = make(g, [cam], **cfg)
    r.forward(p)
    got = view_images(r, 0, C)
    ref = ref_render(g, cam)
    ok = (ref["flags"] & AMBIGUOUS_GRAD) == 0
    assert ok.mean() > 0.9
    for k in ("rgb", "depth", "sem", "T"):
        check_close(k, got[k], ref[k], FWD_REL, FWD_ABS, mask=ok)
    rng = np.random.default_rng(n)
    up = [(rng.normal(size=s) * ok).astype(np.float32) for s in ((3, H, W), (H, W), (C, H, W))]
    grads = {k: torch.zeros_like(v) for k, v in p.items()}
    r.backward(p, grads, dL=tuple(torch.tensor(u.reshape(-1), device="cuda") for u in up))
    want = oracle.render_backward(g, cam, *[u.astype(np.float64) for u in up])
    check_grads({k: v.cpu().numpy() for k, v in grads.items()}, want, KEYS)


@pytest.mark.parametrize("C", [4, 16])
def test_half_mask_lists_with_a_larger_bound_on_the_adjoint_s_pixels(C):
    """Lists with half masks take the half-tile adjoint whatever pixels_per_thread_bwd bounds."""
    test_stacks_around_the_chunk_size_match_oracle(
        17, C, dict(tile_w=8, tile_h=8, pixels_per_thread=1, pixels_per_thread_bwd=2, half_masks=True))


@pytest.mark.parametrize("M, N, K, pad", [(130, 72, 128, 0), (130, 72, 128, 1), (128, 160, 4096, 4), (64, 288, 192, 3),
                                          (300, 32, 64, 2)])
@pytest.mark.parametrize("accumulate", [0, 1])
def test_gemm_epilogue_edges_and_unaligned_rows(M, N, K, pad, accumulate):
    """32-column blocks that end inside or at the matrix, output rows with and without 16-byte
    alignment, stored and accumulated (4-wide reductions): the tolerance of the GEMM tests, and
    nothing written beyond the N columns of a row."""
    import ctypes
    from paper_2412_01217_gb300._lib import call
    torch.manual_seed(M + N + pad)
    A = torch.randn(M, K, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, device="cuda").to(torch.bfloat16)
    D = torch.full((M, N + pad), 0.5, device="cuda")
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    call("sg_gemm_bf16", ptr(A), K, ptr(B), K, M, N, K, ptr(D), N + pad, accumulate, None,
         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    ref = A.double() @ B.double().T + (0.5 if accumulate else 0.0)
    assert (D[:, :N].double() - ref).abs().max().item() <= 1e-5 * ref.abs().max().item() + 1e-3
    assert bool((D[:, N:] == 0.5).all())


@pytest.mark.parametrize("M, N", [(4865, 128), (4865, 100), (9728, 65)])
def test_gemm_with_few_tiles_takes_narrower_ones(M, N):
    """64-column tiles (39 to 76 tiles of 128 columns), with ragged rows and columns: the result
    of each row block computed alone (32-column tiles, the same K order), bit for bit."""
    import ctypes
    from paper_2412_01217_gb300._lib import call
    torch.manual_seed(M + N)
    K = 192
    A = torch.randn(M, K, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, device="cuda").to(torch.bfloat16)
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    D, E = torch.full((M, N), 0.5, device="cuda"), torch.full((M, N), 0.5, device="cuda")
    call("sg_gemm_bf16", ptr(A), K, ptr(B), K, M, N, K, ptr(D), N, 0, None, st)
    for m in range(0, M, 1024):
        a, e = A[m:m + 1024], E[m:m + 1024]
        call("sg_gemm_bf16", ptr(a), K, ptr(B), K, a.shape[0], N, K, ptr(e), N, 0, None, st)
    torch.cuda.synchronize()
    ref = A.double() @ B.double().T
    assert (D.double() - ref).abs().max().item() <= 1e-5 * ref.abs().max().item() + 1e-3
    assert torch.equal(D, E)


def test_mlp_backward_takes_unaligned_targets():
    """The loss head reads Y and the targets 16 bytes at a time only when both are aligned: the
    same batch with targets one float off gives the same bf16 output gradients."""
    from paper_2412_01217_gb300.learned_init import MLPInit
    B = 256
    torch.manual_seed(1)
    X = torch.randn(B, 2048, device="cuda").to(torch.bfloat16)
    buf = torch.randn(B * 32 + 1, device="cuda")
    shifted = buf[1:].view(B, 32)
    out = []
    for T in (shifted, shifted.clone()):
        net = MLPInit(seed=3)
        net.train_step(X, X.T.contiguous(), T, B, torch.zeros(1, device="cuda"))
        a, _ = net.acts(B)
        out.append({k: a[k].clone() for k in ("dY", "dYt", "dH2", "dH1t")})
    for k in out[0]:
        assert torch.equal(out[0][k], out[1][k]), k
