"""The autotuners keep their choices by what selects the kernels: a lattice of another closure kind, or a
batch without a two-step tiling, is timed on its own and not given another's choice."""
import time

import numpy as np
import pytest

from paper_2101_03055_gb300 import inputs as I
from test_parity_gpu import _rand_problem

pytestmark = pytest.mark.gpu


def created_in(make):
    t = time.perf_counter()
    s = make()
    t = time.perf_counter() - t
    s.close()
    return t


def check(make, problems):
    """Every first creation is timed (tuned), every second one is not."""
    first, second = [], []
    for pb in problems:
        first.append(created_in(lambda: make(pb)))
        second.append(min(created_in(lambda: make(pb)) for _ in range(3)))
    for a, b in zip(first, second):
        assert a > 3 * b, (first, second)


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_single_lattice(cdf, storage):
    box = _rand_problem(211, 97, 2, 1, "mixed", "noslip_noflux", force=False)
    forced = _rand_problem(211, 97, 2, 1, "mixed", "noslip_noflux")
    source = forced.replace(skind="const", S=np.array([1e-6, -1e-6]))  # no kind of its own
    cdf.Solver(box.replace(nx=64, ny=64, phi0=box.phi0[:, :64, :64], u0=box.u0[:, :64, :64], p0=box.p0[:64, :64]),
               storage=storage).close()  # the first kernels' loading
    check(lambda pb: cdf.Solver(pb, storage=storage, init=False), [box, forced, source])


def test_batch(cdf):
    wide = [_rand_problem(40, 70, 2, k, "periodic", "noslip_noflux") for k in range(4)]
    plain = [_rand_problem(40, 70, 2, k, "periodic", "noslip_noflux", force=False) for k in range(4)]
    short = [_rand_problem(5, 560, 2, k, "periodic", "noslip_noflux") for k in range(4)]
    assert {sum(p.nodes for p in b) for b in (wide, plain, short)} == {11200}
    cdf.BatchSolver([_rand_problem(20, 20, 2, 1, "periodic", "noslip_noflux")]).close()
    check(lambda pbs: cdf.BatchSolver(pbs, init=False), [wide, plain, short])
