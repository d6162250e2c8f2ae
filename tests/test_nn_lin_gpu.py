"""The convolutions without im2col copies (conv3x3_lin_kernel, conv3x3_wgrad_lin_kernel).

Forward and input gradient run the MMAs of the staged im2col kernels in the same
order, so they give the same bits; the weight and bias gradients are compared
with the FP64 layer oracle.  Their bounds: the products of BF16 values are exact
in FP32 and each of the P sums of a weight is rounded once per product, so the
relative L2 error stays below P 2^-24 for the at most 1024 positions of one split
and the few dozen splits after it (1100 2^-24 = 7e-5 at worst, about its
square root, 2e-6, for random signs; bound 1e-5, as for the other paths).
"""
import math

import numpy as np
import pytest

from oracle import nn_oracle as R

pytestmark = pytest.mark.gpu

# one pixel; one row and one column; sizes around a tile of 128 positions ((H + 1)(W + 1) = 128,
# 126, 130); several tiles with a ragged end; K of 1.1 to 16 ring buffers; every output width;
# 384 channels on rows too wide for the slab (the staged kernels take it)
SHAPES = [(1, 1, 1, 16, 32), (3, 1, 9, 16, 64), (2, 17, 1, 32, 32), (1, 7, 15, 16, 32), (1, 6, 17, 48, 96),
          (1, 12, 9, 32, 160), (2, 31, 33, 96, 32), (5, 13, 40, 64, 128), (1, 16, 16, 896, 32), (3, 8, 8, 256, 256),
          (2, 20, 23, 80, 512), (40, 24, 31, 16, 32), (1, 5, 300, 384, 32), (1, 3, 700, 32, 64)]


@pytest.fixture(scope="module")
def S(cdf):
    import torch
    from paper_2101_03055_gb300 import surrogate
    surrogate.nn_lib()
    return surrogate, torch


def make(torch, N, H, W, cin, cout):
    g = torch.Generator(device="cuda").manual_seed(N + H * W + cin + cout)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    bf = torch.bfloat16
    return (r(N, H, W, cin).to(bf), (r(cout, 3, 3, cin) / math.sqrt(9 * cin)).to(bf), r(cout),
            r(N, H, W, cout).to(bf))


@pytest.mark.parametrize("N,H,W,cin,cout", SHAPES)
def test_same_bits_as_staged_kernels(S, N, H, W, cin, cout):
    sur, torch = S
    x, w, b, dy = make(torch, N, H, W, cin, cout)
    got = {}
    try:
        for path in (1, 2):
            sur.set_tensor_path(path)
            got[path] = [sur.conv3x3_fwd(x, w, b, True), sur.conv3x3_fwd(x, w, None, False),
                         sur.conv3x3_bwd_data(dy, w, cin)]
        for a, c in zip(got[1], got[2]):
            assert torch.equal(a, c)
    finally:
        sur.set_tensor_path(True)
    assert sur.tensor_error_flag() == 0


@pytest.mark.parametrize("N,H,W,cin,cout", [s for s in SHAPES if s[0] * s[1] * s[2] * s[3] * s[4] < 3e8])
def test_weight_gradient(S, N, H, W, cin, cout):
    sur, torch = S
    x, _, _, dy = make(torch, N, H, W, cin, cout)
    dw = torch.full((cout, 3, 3, cin), 0.5, device="cuda")
    db = torch.full((cout,), -0.25, device="cuda")
    sur.conv3x3_bwd_weight(x, dy, dw, db)
    wr, br = R.conv3x3_bwd_weight(x.double().cpu().numpy(), dy.double().cpu().numpy())
    rel = lambda a, c: float(np.linalg.norm(a - c) / np.linalg.norm(c))  # noqa: E731
    assert rel(dw.double().cpu().numpy(), wr + 0.5) < 1e-5  # added to what was there
    assert rel(db.double().cpu().numpy(), br - 0.25) < 1e-5
    assert sur.tensor_error_flag() == 0


def test_weights_behind_an_offset(S):
    """Weights 16 bytes into their allocation (the least alignment the copies take)."""
    sur, torch = S
    x, w, b, _ = make(torch, 1, 9, 11, 16, 32)
    base = torch.empty(w.numel() + 8, dtype=torch.bfloat16, device="cuda")
    shifted = base[8:].view(w.shape)
    shifted.copy_(w)
    assert torch.equal(sur.conv3x3_fwd(x, shifted, b, True), sur.conv3x3_fwd(x, w, b, True))
