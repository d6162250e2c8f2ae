"""One step per launch: which closure kind's kernel runs depends on the lattice's size, the bits do
not, and a kind's lattice is not slower than one for which every term is decided at run time."""
import numpy as np
import pytest

from paper_2101_03055_gb300 import inputs as I
from test_parity_gpu import _rand_problem

pytestmark = pytest.mark.gpu


# on either side of 250,000 nodes (forced kind) and of 100 MB of populations, 689,853 nodes (both)
@pytest.mark.parametrize("nx,ny", [(500, 499), (500, 500), (830, 831), (831, 831)])
@pytest.mark.parametrize("flow", ["forced", "plume"])
@pytest.mark.parametrize("block", [(128, 1), (224, 0)])
def test_same_bits_as_two_steps_a_launch(cdf, nx, ny, flow, block):
    pb = I.chemotaxis_plume(nx, ny) if flow == "plume" else _rand_problem(nx, ny, 2, 3, "mixed", "noslip_noflux")
    out = []
    for kw in (dict(temporal=-1, resident=-1, block=block), dict(temporal=1, resident=-1, temporal_shape=(32, 8, 14))):
        s = cdf.Solver(pb, **kw)
        s.step(4)
        out.append(s.moments())
        s.close()
    assert np.array_equal(*out)


def step_ms(torch, s, n=64):
    s.step(n)
    torch.cuda.synchronize()
    best = 1e9
    for _ in range(5):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        s.step(n)
        s.step(n)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


@pytest.mark.parametrize("nx,ny", [(96, 96), (200, 150)])
def test_forced_kind_is_not_slower(cdf, nx, ny):
    """Against a constant source, which has no kind of its own; the forced kind's kernels took 1.29 and 1.23
    times its time."""
    import torch
    forced = _rand_problem(nx, ny, 2, 3, "mixed", "noslip_noflux")
    t = []
    for pb in (forced, forced.replace(skind="const", S=np.array([1e-6, -1e-6]))):
        s = cdf.Solver(pb, temporal=-1, resident=-1, block=(128, 1))
        t.append(step_ms(torch, s))
        s.close()
    assert t[0] <= 1.1 * t[1], t
