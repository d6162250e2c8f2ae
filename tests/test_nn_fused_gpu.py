"""The small layers at both access widths (8 channels a thread, or one where a count is no multiple
of 8) and the fused layers of the network's passes.

Pooling, upsampling, copies and masks are compared bit for bit with the same operations in
PyTorch (one BF16 rounding of FP32 sums of at most four BF16 values, which FP32 adds exactly or
in the same order); the fused calls with the separate calls they stand for, bit for bit; the head's
FP32 sums of up to C terms within C 2^-24 relative, loosely 1e-5."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S(cdf):
    import torch
    from paper_2101_03055_gb300 import surrogate
    surrogate.nn_lib()
    return surrogate, torch


def rand(torch, seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)


def relu_like(torch, seed, *shape):
    return rand(torch, seed, *shape).relu()


@pytest.mark.parametrize("N,H,W,C", [(1, 2, 2, 8), (2, 6, 10, 12), (3, 4, 14, 40), (1, 2, 2, 1), (5, 8, 6, 24)])
def test_small_layers_at_both_widths(S, N, H, W, C):
    sur, torch = S
    x = rand(torch, 1, N, H, W, C)
    q = x.float().view(N, H // 2, 2, W // 2, 2, C)
    assert torch.equal(sur.avgpool2_fwd(x), (0.25 * (((q[:, :, 0, :, 0] + q[:, :, 0, :, 1]) + q[:, :, 1, :, 0])
                                                    + q[:, :, 1, :, 1])).to(torch.bfloat16))
    up = lambda t: t.repeat_interleave(2, 1).repeat_interleave(2, 2)  # noqa: E731
    assert torch.equal(sur.avgpool2_bwd(x, 2 * H, 2 * W), up((0.25 * x.float()).to(torch.bfloat16)))
    y = rand(torch, 2, N, 2 * H, 2 * W, C + 8)
    want = y.clone()
    want[..., 8:] = up(x)
    sur.upsample2_into(x, y, 8)
    assert torch.equal(y, want)
    v = y[..., 8:].float().view(N, H, 2, W, 2, C)
    s = ((v[:, :, 0, :, 0] + v[:, :, 0, :, 1]) + v[:, :, 1, :, 0]) + v[:, :, 1, :, 1]
    assert torch.equal(sur.upsample2_bwd_from(y, C, 8), s.to(torch.bfloat16))
    z = rand(torch, 3, N, H, W, C + 8)
    want = z.clone()
    want[..., 8:] = (want[..., 8:].float() + x.float()).to(torch.bfloat16)
    sur.copy_channels(x, z, 0, 8, C, accumulate=True)
    assert torch.equal(z, want)
    d, m = rand(torch, 4, N, H, W, C), relu_like(torch, 5, N, H, W, C)
    want = torch.where(m > 0, d, torch.zeros_like(d))
    sur.relu_bwd(d, m)
    assert torch.equal(d, want)


@pytest.mark.parametrize("P,C,O", [(1, 8, 1), (63, 12, 4), (513, 32, 4), (2049, 40, 7)])
def test_head(S, P, C, O):
    sur, torch = S
    x = relu_like(torch, 6, 1, 1, P, C)
    g = torch.Generator(device="cuda").manual_seed(7)
    w, b = torch.randn((O, C), generator=g, device="cuda"), torch.randn(O, generator=g, device="cuda")
    dout = torch.randn((1, 1, P, O), generator=g, device="cuda")
    rel = lambda a, c: float((a.double() - c).norm() / c.norm())  # noqa: E731
    assert rel(sur.head_fwd(x, w, b), x.double() @ w.double().T + b.double()) < 1e-5
    dw, db = torch.zeros_like(w), torch.zeros_like(b)
    dx = sur.head_bwd(x, w, dout, dw, db)
    d2, x2 = dout.double().view(P, O), x.double().view(P, C)
    assert rel(dw, d2.T @ x2) < 1e-5 and rel(db, d2.sum(0)) < 1e-5
    assert rel(dx.view(P, C), d2 @ w.double()) < 4e-3  # one BF16 rounding, 2^-9 a value
    masked = sur.head_bwd_relu(x, w, dout, torch.zeros_like(w), torch.zeros_like(b))
    assert torch.equal(masked, torch.where(x > 0, dx, torch.zeros_like(dx)))


@pytest.mark.parametrize("N,H,W,C,Cs", [(1, 2, 2, 8, 16), (2, 4, 6, 32, 16), (3, 6, 2, 12, 20)])
def test_fused_layers_equal_their_parts(S, N, H, W, C, Cs):
    sur, torch = S
    x, skip = relu_like(torch, 8, N, H, W, C), relu_like(torch, 9, N, 2 * H, 2 * W, Cs)
    cat = torch.empty((N, 2 * H, 2 * W, C + Cs), dtype=torch.bfloat16, device="cuda")
    sur.upsample2_into(x, cat, 0)
    sur.copy_channels(skip, cat, 0, C, Cs)
    assert torch.equal(sur.upsample2_concat(x, skip), cat)
    dcat = rand(torch, 10, N, 2 * H, 2 * W, C + Cs)
    want = sur.upsample2_bwd_from(dcat, C, 0)
    sur.relu_bwd(want, x)
    assert torch.equal(sur.upsample2_bwd_relu(dcat, x), want)
    dp = rand(torch, 11, N, H, W, Cs)
    want = sur.avgpool2_bwd(dp, 2 * H, 2 * W)
    sur.copy_channels(dcat, want, C, 0, Cs, accumulate=True)
    sur.relu_bwd(want, skip)
    assert torch.equal(sur.pool_skip_bwd_relu(dp, dcat, skip), want)


# the last two: a mask off the kernel's 16 bytes, and rows too wide for it (staged kernels, then the mask)
@pytest.mark.parametrize("N,H,W,cin,cout,shift", [(2, 9, 13, 16, 32, 0), (1, 5, 7, 96, 64, 0), (1, 16, 16, 256, 64, 0),
                                                  (1, 4, 5, 32, 32, 1), (1, 2, 300, 32, 384, 0)])
def test_masked_input_gradient(S, N, H, W, cin, cout, shift):
    sur, torch = S
    dy, w = rand(torch, 12, N, H, W, cout), rand(torch, 13, cout, 3, 3, cin)
    y = relu_like(torch, 14, N * H * W * cin + 8)[shift:shift + N * H * W * cin].view(N, H, W, cin)
    want = sur.conv3x3_bwd_data(dy, w, cin)
    sur.relu_bwd(want, y)
    assert torch.equal(sur.conv3x3_bwd_data_relu(dy, w, y), want)
    assert sur.tensor_error_flag() == 0
