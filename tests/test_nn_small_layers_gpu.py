"""The small layers on channel counts without 16-byte accesses, and on layers too small to fill the chip."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S(cdf):
    import torch
    from paper_2101_03055_gb300 import surrogate
    surrogate.nn_lib()
    return surrogate, torch


def rand(torch, *shape):
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    return torch.randn(shape, generator=g, device="cuda")


def seconds(torch, f):
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        f()
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            for _ in range(20):
                f()
        g.replay()
        best = 1e9
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record(st)
            g.replay()
            e[1].record(st)
            st.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("P,Cx,Cy,src,dst,count", [(1, 1, 1, 0, 0, 1), (257, 33, 40, 0, 7, 33), (1000, 16, 24, 3, 8, 8),
                                                   (333, 24, 32, 8, 16, 16)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_copy_channels(S, P, Cx, Cy, src, dst, count, accumulate):
    """Bit for bit: one BF16 rounding of an exact FP32 sum."""
    sur, torch = S
    x, y = rand(torch, 1, 1, P, Cx).to(torch.bfloat16), rand(torch, 1, 1, P, Cy).to(torch.bfloat16)
    want = y.clone()
    part = x[..., src:src + count].float()
    want[..., dst:dst + count] = (part + want[..., dst:dst + count].float() if accumulate else part).to(torch.bfloat16)
    sur.copy_channels(x, y, src, dst, count, accumulate=accumulate)
    assert torch.equal(y, want)
