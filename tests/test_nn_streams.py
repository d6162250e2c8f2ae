"""Weight gradients at work at the same time, on several streams or from several threads, have
partial sums of their own."""
import pytest


def test_calls_at_work_do_not_share_a_workspace(monkeypatch):
    """A second call that begins before the first has ended (here: inside it) gets another buffer."""
    import torch
    from paper_2101_03055_gb300 import surrogate as S
    used = []

    def gradient(n):
        z = lambda *s: torch.zeros(s)  # noqa: E731
        S.conv3x3_bwd_weight(z(1, n, n, 16), z(1, n, n, 32), z(32, 3, 3, 16), z(32))

    def call(name, *args):
        start = args[9]
        used.append((start, start + args[10]))
        if len(used) < 3:
            gradient(8)

    monkeypatch.setattr(S, "_call", call)
    monkeypatch.setattr(S, "_stream", lambda: None)
    gradient(8)
    used.sort()
    assert len(used) == 3 and all(a[1] <= b[0] for a, b in zip(used, used[1:])), used


@pytest.mark.gpu
def test_two_streams_give_the_serial_bits(cdf):
    import torch
    from paper_2101_03055_gb300 import surrogate as S
    S.nn_lib()
    g = torch.Generator(device="cuda").manual_seed(2)
    shapes = [(4, 64, 64, 64, 64), (2, 96, 96, 32, 32)]
    data = [(torch.randn((n, h, w, ci), generator=g, device="cuda").to(torch.bfloat16),
             torch.randn((n, h, w, co), generator=g, device="cuda").to(torch.bfloat16)) for n, h, w, ci, co in shapes]

    def gradient(k):
        x, dy = data[k]
        dw = torch.zeros((dy.shape[3], 3, 3, x.shape[3]), device="cuda")
        db = torch.zeros(dy.shape[3], device="cuda")
        S.conv3x3_bwd_weight(x, dy, dw, db)
        return dw, db

    want = [gradient(0), gradient(1)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for _ in range(40):
        for k in (0, 1):
            with torch.cuda.stream(streams[k]):
                got.append((k, gradient(k)))
    torch.cuda.synchronize()
    for k, r in got:
        assert torch.equal(r[0], want[k][0]) and torch.equal(r[1], want[k][1])
