"""Both reductions of the decoder gradient's per-block shares (one kernel up to 1024 of them, two
levels beyond), and the GEMM's 64-column tiles against its 128-column ones."""
import ctypes as C

import pytest
import torch

import synthetic
from helpers import check_close
from test_gpu_parity import f32_camera

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [4, 8, 40])
@pytest.mark.parametrize("W, H", [(512, 512), (512, 513), (700, 400)])  # 1024, 1026 and 1094 blocks
def test_decoder_gradient_of_many_blocks(W, H, K):
    """Against 64 bits, with the tolerance of the loss parity test (a square decoder runs on the
    CUDA cores, a block per 256 pixels)."""
    from paper_2412_01217_gb300 import LossConfig, PyramidRasterizer
    cam = f32_camera(synthetic.make_camera(W, H, float(W), float(W), W / 2 - 0.5, H / 2 - 0.5))
    r = PyramidRasterizer(1, K, [cam], 1, loss_cfg=LossConfig(n_classes=K))
    g = torch.Generator(device="cuda").manual_seed(W + H + K)
    P = r.P
    rnd = lambda *s: torch.rand(*s, generator=g, device="cuda")
    sem = torch.randn(K, P, generator=g, device="cuda")
    label = torch.randint(-1, K, (P,), generator=g, device="cuda").int()
    dec, start = 0.5 * torch.randn(K, K, generator=g, device="cuda"), torch.randn(K, K, generator=g, device="cuda")
    dgrad = start.clone()
    r.loss(dict(rgb=rnd(3 * P), depth=rnd(P) + 1, label=label), rendered=(rnd(3 * P), rnd(P) + 1, sem.reshape(-1)),
           decoder=dec, decoder_grad=dgrad)
    torch.cuda.synchronize()
    d = dec.double().requires_grad_(True)
    valid = label >= 0
    z = (d @ sem.double())[:, valid].T
    want, = torch.autograd.grad(torch.nn.functional.cross_entropy(z, label[valid].long()), d)
    check_close("dL/ddecoder", dgrad.cpu().numpy(), (start.double() + want).cpu().numpy(), 1e-4, 1e-6)
    # (the increment alone: the buffer's own rounding aside)
    check_close("increment", (dgrad - start).cpu().numpy(), want.cpu().numpy(), 1e-4, 1e-6)


@pytest.mark.parametrize("M, N", [(4865, 128), (4865, 100), (9728, 65)])
def test_64_column_tiles_give_the_128_column_ones_bits(M, N):
    """39 to 76 row blocks take 64-column tiles; the same rows twice over, 128-column ones."""
    from paper_2412_01217_gb300._lib import call
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = (M + 127) // 128
    assert 4 * blocks > sms and 2 * blocks <= sms < 4 * blocks
    torch.manual_seed(M + N)
    K = 192
    rows = 128 * blocks
    A = torch.randn(rows, K, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, device="cuda").to(torch.bfloat16)
    p = lambda t: C.c_void_p(t.data_ptr())
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    two = torch.cat([A, A])
    D, E = torch.full((M, N), 0.5, device="cuda"), torch.full((2 * rows, N), 0.5, device="cuda")
    call("sg_gemm_bf16", p(A), K, p(B), K, M, N, K, p(D), N, 0, None, st)
    call("sg_gemm_bf16", p(two), K, p(B), K, 2 * rows, N, K, p(E), N, 0, None, st)
    torch.cuda.synchronize()
    assert torch.equal(D, E[:M]) and torch.equal(E[:rows], E[rows:])
