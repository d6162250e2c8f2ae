"""The weight gradient's workspace holds every launch of a call: batches of 2^30 padded
positions and more run in several, the last one with fewer images and a tiling of its own."""
import pytest


@pytest.mark.parametrize("H,W", [(4095, 4095), (2999, 5003)])
@pytest.mark.parametrize("cin,cout", [(16, 32), (32, 32), (64, 128), (256, 256)])
def test_covers_the_remainder(H, W, cin, cout):
    from paper_2101_03055_gb300 import surrogate
    ws = surrogate.nn_lib().cdf_nn_conv3x3_bwd_weight_workspace
    images = ((1 << 30) - 1) // ((H + 1) * (W + 1))
    for r in range(1, images):
        assert ws(images + r, H, W, cin, cout) >= max(ws(r, H, W, cin, cout), ws(images, H, W, cin, cout))
