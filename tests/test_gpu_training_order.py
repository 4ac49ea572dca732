"""The training step of the learned initializer gives the same bits every time: the parts of the
K-split weight gradients and of the loss are added in a fixed order, not atomically.  And the
sums are the ones the unordered entry point forms: each weight gradient within the rounding of
its parts' sum."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


def _batch(B, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(B, 2048, generator=g, device="cuda") * 0.5
    X[:, 2009:] = 0
    X = X.to(torch.bfloat16)
    return X, X.T.contiguous(), torch.randn(B, 32, generator=g, device="cuda")


@pytest.mark.parametrize("B", [128, 640, 4096, 16384])
def test_steps_are_reproducible(B):
    """B = 128 is two K chunks (two splits each), 640 ten; 16384 is split 19 and 64 ways."""
    from paper_2412_01217_gb300.learned_init import MLPInit
    X, Xt, T = _batch(B, B)
    runs = []
    for _ in range(4):
        net, loss = MLPInit(seed=2), torch.zeros(1, device="cuda")
        for _ in range(3):
            net.train_step(X, Xt, T, B, loss)
        torch.cuda.synchronize()
        assert int(net.status.item()) == 0
        runs.append([t.clone() for t in (*net.params, *net.m, *net.v, loss)])
    for r in runs[1:]:
        for a, b in zip(r, runs[0]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("B", [128, 2560, 16384])
@pytest.mark.parametrize("start", [0.0, 0.5])
def test_ordered_sums_match_the_unordered(B, start):
    """Both add the same FP32 parts (at most 64) to what the buffers hold; an addition is off by
    at most 2^-24 of its result, so a gradient by at most 65 x 2^-24 of the sum of |parts| and
    |start|.  The parts' absolute sum is at most sum_k |a_k b_k|."""
    from paper_2412_01217_gb300._lib import SgMlpGrads, call
    from paper_2412_01217_gb300.learned_init import MLPInit
    p = lambda t: C.c_void_p(t.data_ptr())
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    net = MLPInit(seed=2)
    X, Xt, T = _batch(B, B + 1)
    net.forward(X, B)
    a, s = net.acts(B)
    got = []
    for ordered in (False, True):
        g = [torch.full_like(t, start) for t in net.params]
        G, loss, n = SgMlpGrads(*[t.data_ptr() for t in g]), torch.full((1,), start, device="cuda"), net.net()
        head = (C.byref(n), p(Xt), p(T), p(net.out_w), B, C.byref(s), C.byref(G), p(loss))
        if ordered:
            work = torch.full_like(net.work(B), 0xff)  # (NaN: every part is written)
            call("sg_mlp_backward_ordered", *head, p(work), work.numel(), p(net.status), st)
        else:
            call("sg_mlp_backward", *head, p(net.status), st)
        torch.cuda.synchronize()
        got.append([*g, loss])
    assert int(net.status.item()) == 0
    f = lambda k: a[k].double().abs()
    sums = (f("dH1t") @ X.double().abs(), f("dH2t") @ f("H1"), f("dYt") @ f("H2"))
    for u, o, bound in zip(got[0], got[1], sums):
        assert bool(((u.double() - o.double()).abs() <= 65 * 2.0 ** -24 * (bound + start) * 2).all())
    for u, o in zip(got[0][3:6], got[1][3:6]):
        assert torch.equal(u, o)  # bias gradients: one kernel for both
    assert got[1][6].item() == pytest.approx(got[0][6].item(), rel=1e-5)


def test_ordered_backward_checks_its_workspace():
    from paper_2412_01217_gb300._lib import SgError, SgMlpGrads, call
    from paper_2412_01217_gb300.learned_init import MLPInit
    B = 256
    net = MLPInit(seed=2)
    X, Xt, T = _batch(B, 3)
    net.forward(X, B)
    _, s = net.acts(B)
    n, G, work, loss = net.net(), SgMlpGrads(*[t.data_ptr() for t in net.grads]), net.work(B), torch.zeros(1, device="cuda")
    p = lambda t: C.c_void_p(t.data_ptr())
    head = (C.byref(n), p(Xt), p(T), p(net.out_w), B, C.byref(s), C.byref(G), p(loss))
    for ptr, size, code in ((p(work), work.numel() - 1, 2), (None, work.numel(), 1),
                            (C.c_void_p(work.data_ptr() + 4), work.numel(), 1)):
        with pytest.raises(SgError) as e:
            call("sg_mlp_backward_ordered", *head, ptr, size, p(net.status), None)
        assert e.value.code == code
    torch.cuda.synchronize()
    assert all(bool((t == 0).all()) for t in net.grads)
