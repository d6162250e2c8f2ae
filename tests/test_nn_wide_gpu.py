"""Convolutions on wide images: whichever kernel the default path takes, the bits are those of
the two-buffer im2col kernel (path 2: the same MMAs in the same order), and it is not slower than
that kernel."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S(cdf):
    import torch
    from paper_2101_03055_gb300 import surrogate
    surrogate.nn_lib()
    return surrogate, torch


def make(torch, N, H, W, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(H * W + cin)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    bf = torch.bfloat16
    return (r(N, H, W, cin).to(bf), (r(cout, 3, 3, cin) / math.sqrt(9 * cin)).to(bf), r(cout), r(N, H, W, cout).to(bf))


def on_path(S, path, f):
    S.set_tensor_path(path)
    try:
        return f()
    finally:
        S.set_tensor_path(True)


# rows of one and of several 128-pixel tiles, at each of its channel counts and output widths, one
# image row, more tiles than CTAs, and widths on either side of each kernel's range
SHAPES = [(1, 3, 128, 16, 32), (2, 1, 384, 64, 64), (1, 5, 640, 64, 32), (3, 2, 1024, 32, 128), (1, 40, 2048, 16, 64),
          (1, 7, 1536, 32, 96), (1, 300, 512, 64, 256), (1, 9, 3328, 16, 32), (1, 3, 299, 32, 32), (1, 3, 300, 32, 32),
          (1, 30, 1500, 32, 32), (1, 60, 752, 64, 64), (1, 40, 200, 192, 64), (1, 128, 128, 256, 256), (1, 65, 71, 384, 128)]


@pytest.mark.parametrize("shape", SHAPES)
def test_same_bits_as_im2col(S, shape):
    S, torch = S
    x, w, b, dy = make(torch, *shape)
    for f in (lambda: S.conv3x3_fwd(x, w, b, True), lambda: S.conv3x3_fwd(x, w, None, False),
              lambda: S.conv3x3_bwd_data(dy, w, shape[3]),
              lambda: S.conv3x3_bwd_data_relu(dy, w, x)):
        got, want = f(), on_path(S, 2, f)
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    assert S.tensor_error_flag() == 0


def seconds(torch, f):
    for _ in range(3):
        f()
    best = 1e9
    for _ in range(5):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(5):
            f()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("shape,forward,factor", [
    ((1, 682, 1536, 32, 32), True, 0.7), ((1, 512, 2048, 32, 32), True, 0.7), ((1, 655, 3200, 16, 32), True, 0.7),
    ((1, 512, 1024, 64, 64), True, 0.7), ((1, 697, 752, 64, 64), True, 1.3), ((1, 697, 752, 64, 64), False, 1.3),
    ((1, 1310, 1600, 16, 32), False, 1.3), ((1, 124, 700, 192, 64), False, 1.3)])
def test_time_against_im2col(S, shape, forward, factor):
    """Rows whose halo outweighs the tile took up to 18 times the im2col kernel's time; rows of whole
    128-pixel tiles with 16, 32 or 64 input channels have a kernel that takes half of it, forward."""
    S, torch = S
    x, w, b, dy = make(torch, *shape)
    f = (lambda: S.conv3x3_fwd(x, w, b, True)) if forward else (lambda: S.conv3x3_bwd_data(dy, w, shape[3]))
    assert seconds(torch, f) <= factor * on_path(S, 2, lambda: seconds(torch, f))
