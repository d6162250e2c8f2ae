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


@pytest.mark.parametrize("P,C,O", [(1, 7, 1), (257, 33, 5), (1000, 12, 9), (300, 32, 5), (262143, 9, 3), (262144, 9, 3),
                                   (262200, 5, 1)])
def test_head_fwd(S, P, C, O):
    """FP32 sums of at most 33 products, 33 2^-24 of the terms' absolute sum."""
    sur, torch = S
    x, w, b = rand(torch, 1, 1, P, C).to(torch.bfloat16), rand(torch, O, C), rand(torch, O)
    got = sur.head_fwd(x, w, b).double().view(P, O)
    x2, w2 = x.double().view(P, C), w.double()
    bound = (x2.abs() @ w2.abs().T + b.double().abs()) * (34 * 2.0 ** -24)
    assert bool(((got - (x2 @ w2.T + b.double())).abs() <= bound).all())


def test_head_fwd_on_odd_channels_is_not_slower(S):
    """33 channels on 64 x 64 pixels took 1.44 times the time of 32 with four outputs a thread."""
    sur, torch = S
    t = []
    for C in (33, 32):
        x, w, b = rand(torch, 1, 64, 64, C).to(torch.bfloat16), rand(torch, 5, C), rand(torch, 5)
        t.append(seconds(torch, lambda: sur.head_fwd(x, w, b)))
    assert t[0] <= 1.2 * t[1]


@pytest.mark.parametrize("n", [1, 255, 257, 5120, 38912, 38913, 40959, 100001])
def test_mse(S, n):
    """The gradient bit for bit; the loss within its FP32 rounding: three roundings a term and chains
    below 300 additions of positive terms."""
    sur, torch = S
    p, t = rand(torch, 2, n)
    loss, grad = sur.mse(p, t)
    want = ((p.double() - t.double()) ** 2).mean()
    assert torch.equal(grad, 2.0 * (p - t) / torch.full_like(p, n))  # (by a tensor: an IEEE quotient)
    assert abs(float(loss) / float(want) - 1) <= 303 * 2.0 ** -24


def test_mse_of_few_values_fills_the_chip(S):
    """5120 values, eight a thread, took 1.9 times the time of 64."""
    sur, torch = S
    a, b = rand(torch, 5120), rand(torch, 64)
    assert seconds(torch, lambda: sur.mse(a, a)) <= 1.5 * seconds(torch, lambda: sur.mse(b, b))
