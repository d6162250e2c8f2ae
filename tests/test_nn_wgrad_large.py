"""The weight gradient where one launch cannot take every split of the positions: its
workspace stays bounded, and with it the rows of a launch's grid (a row is a split of at
least 36 x 16 x 32 bytes, and a grid has at most 65,535)."""
import pytest

BOUND = 192 << 20  # 160 MiB of partial sums, at least one split, and the bias gradient's


@pytest.mark.parametrize("N,H,W,cin,cout", [(16, 256, 256, 256, 256), (16, 512, 512, 256, 256), (64, 1024, 1024, 16, 32),
                                            (1024, 256, 256, 32, 32), (1, 8192, 8192, 16, 32), (70, 1000, 1000, 16, 32),
                                            (63, 4095, 4095, 16, 32), (200, 4095, 4095, 64, 64), (1, 30000, 30000, 32, 64)])
def test_workspace_is_bounded(N, H, W, cin, cout):
    from paper_2101_03055_gb300 import surrogate
    got = surrogate.nn_lib().cdf_nn_conv3x3_bwd_weight_workspace(N, H, W, cin, cout)
    assert 36 * cin * cout <= got <= BOUND


def _check(S, torch, N, H, W, cin, cout, seed):
    """dw and db against FP64 sums, image by image; the FP32 sums of 1024 positions, of the splits of
    a launch and of the launches each keep the relative error near the square root of their
    length times 2^-24, below 1e-5 together (the bound of the other paths)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty((N, H, W, cin), device="cuda", dtype=torch.bfloat16)
    dy = torch.empty((N, H, W, cout), device="cuda", dtype=torch.bfloat16)
    for n in range(N):
        x[n] = torch.randn((H, W, cin), generator=g, device="cuda")
        dy[n] = torch.randn((H, W, cout), generator=g, device="cuda")
    out = []
    for _ in range(2):
        dw = torch.full((cout, 3, 3, cin), 0.5, device="cuda")
        db = torch.full((cout,), 0.25, device="cuda")
        S.conv3x3_bwd_weight(x, dy, dw, db)
        out.append((dw, db))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    want_w = torch.zeros((3, 3, cout, cin), device="cuda", dtype=torch.float64)
    want_b = torch.zeros(cout, device="cuda", dtype=torch.float64)
    for n in range(N):
        xp = torch.nn.functional.pad(x[n].double(), (0, 0, 1, 1, 1, 1))
        d = dy[n].double().reshape(-1, cout)
        want_b += d.sum(0)
        for ky in range(3):
            for kx in range(3):
                want_w[ky, kx] += d.T @ xp[ky:ky + H, kx:kx + W].reshape(-1, cin)
    want_w = want_w.permute(2, 0, 1, 3)
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())  # noqa: E731
    assert rel(out[0][0] - 0.5, want_w) <= 1e-5
    assert rel(out[0][1] - 0.25, want_b) <= 1e-5
    assert S.tensor_error_flag() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(5, 100, 131, 256, 256), (16, 128, 128, 256, 256), (1, 211, 300, 16, 32 * 96),
                                   (64, 1024, 1024, 16, 32)])
def test_several_launches(cdf, shape):
    import torch
    from paper_2101_03055_gb300 import surrogate as S
    S.nn_lib()
    _check(S, torch, *shape, seed=sum(shape))


@pytest.mark.parametrize("N,H,W", [(1, 33000, 33000), (3, 40000, 40000), (2, 5, 1 << 28)])
def test_large_images_run_on_the_tensor_cores(N, H, W):
    """An image of 2^30 positions and more goes in bands of rows; a workspace of 4 bytes would
    mean the warp-level kernel."""
    from paper_2101_03055_gb300 import surrogate
    got = surrogate.nn_lib().cdf_nn_conv3x3_bwd_weight_workspace(N, H, W, 16, 32)
    assert (got == 4) if W == 1 << 28 else 36 * 16 * 32 <= got <= BOUND


@pytest.mark.gpu
def test_bands_of_a_large_image(cdf):
    """33000 x 33000 pixels, zero but for the first and last rows and those on either side of the
    bands' edge: the sums of those rows."""
    import torch
    from paper_2101_03055_gb300 import surrogate as S
    S.nn_lib()
    H = W = 33000
    if torch.cuda.mem_get_info()[0] < 130 << 30:
        pytest.skip("needs 105 GB on the device")
    edge = ((1 << 30) - 1) // (W + 1) - 3
    rows = [*range(0, 3), *range(edge - 3, edge + 3), *range(H - 3, H)]
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.zeros((1, H, W, 16), device="cuda", dtype=torch.bfloat16)
    dy = torch.zeros((1, H, W, 32), device="cuda", dtype=torch.bfloat16)
    for y in rows:
        x[0, y] = torch.randn((W, 16), generator=g, device="cuda")
        dy[0, y] = torch.randn((W, 32), generator=g, device="cuda")
    dw, db = torch.zeros((32, 3, 3, 16), device="cuda"), torch.zeros(32, device="cuda")
    S.conv3x3_bwd_weight(x, dy, dw, db)
    want_w, want_b = torch.zeros((3, 3, 32, 16), device="cuda", dtype=torch.float64), 0
    for y in rows:
        d = dy[0, y].double()
        want_b = want_b + d.sum(0)
        for ky in range(3):
            if 0 <= y + ky - 1 < H:
                xp = torch.nn.functional.pad(x[0, y + ky - 1].double(), (0, 0, 1, 1))
                for kx in range(3):
                    want_w[ky, kx] += d.T @ xp[kx:kx + W]
    want_w = want_w.permute(2, 0, 1, 3)
    assert float((dw.double() - want_w).norm() / want_w.norm()) <= 1e-5
    assert float((db.double() - want_b).norm() / want_b.norm()) <= 1e-5
    assert S.tensor_error_flag() == 0


@pytest.mark.gpu
def test_warp_level_kernel_on_many_pixels(cdf):
    """More pixels than 65,535 splits of 4096, zero but for a few rows."""
    import torch
    from paper_2101_03055_gb300 import surrogate as S
    S.nn_lib()
    H, W = 8200, 33000
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 26 GB on the device")
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.zeros((1, H, W, 16), device="cuda", dtype=torch.bfloat16)
    dy = torch.zeros((1, H, W, 32), device="cuda", dtype=torch.bfloat16)
    for y in (0, 4000, H - 1):
        x[0, y] = torch.randn((W, 16), generator=g, device="cuda")
        dy[0, y] = torch.randn((W, 32), generator=g, device="cuda")
    got = []
    for path in (1, 0):
        dw, db = torch.zeros((32, 3, 3, 16), device="cuda"), torch.zeros(32, device="cuda")
        S.set_tensor_path(path)
        try:
            S.conv3x3_bwd_weight(x, dy, dw, db)
        finally:
            S.set_tensor_path(True)
        got.append((dw.double(), db.double()))
    for a, b in zip(*got):  # both within 1e-5 of the exact sums
        assert float((a - b).norm() / a.norm()) <= 2e-5


def test_workspace_off_16_bytes_is_refused():
    """The check comes before any launch: the addresses here are never used."""
    from paper_2101_03055_gb300 import surrogate as S
    L = S.nn_lib()
    for ws in (0x10004, 0x10008):
        assert L.cdf_nn_conv3x3_bwd_weight(0x1000, 0x2000, 0x3000, None, 1, 8, 8, 16, 32, ws, 1 << 30, None) != 0
        assert b"16 bytes" in L.cdf_nn_last_error()
