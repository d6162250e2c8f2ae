"""Whole-batch launches of two steps (step2_batch_kernel) and the one-launch
initialisation and packing: every instance bit for bit the single-lattice solver.

Sizes where the tiling can go wrong: lattices smaller than one tile, one node or
row more than a tile, one row, a periodic axis of exactly the region's width, of
6 nodes (the smallest tiling) and of 5 (the persistent kernel takes the batch)."""
import numpy as np
import pytest

from test_parity_gpu import _rand_problem

pytestmark = pytest.mark.gpu


def check(cdf, pbs, steps=(1, 2, 35, 3)):
    import torch
    b = cdf.BatchSolver(pbs, tile=(64, 4), mode=0, init=False)
    m = pbs[0].m
    stacks = [np.concatenate([pb.phi0.reshape(m, pb.ny, pb.nx), pb.u0.reshape(2, pb.ny, pb.nx),
                              pb.p0.reshape(1, pb.ny, pb.nx)]).astype(np.float32) for pb in pbs]
    b.init_moments_device(torch.from_numpy(np.concatenate([s.ravel() for s in stacks])).cuda())
    for n in steps:
        b.step(n)
    out = torch.empty(b.stack_floats(), dtype=torch.float32, device="cuda")
    b.moments_device(out)
    got, off = out.cpu().numpy().astype(np.float64), 0
    for pb, st in zip(pbs, stacks):
        s = cdf.Solver(pb, init=False, temporal=-1, resident=-1, block=(128, 1))
        s.init_moments_device(torch.from_numpy(st).cuda())
        for n in steps:
            s.step(n)
        want = s.moments()
        assert np.array_equal(got[off:off + want.size].reshape(want.shape), want), (pb.nx, pb.ny)
        off += want.size


@pytest.mark.parametrize("m", [1, 2, 3, 4])
@pytest.mark.parametrize("xcase,ycase", [("periodic", "periodic"), ("mixed", "freeslip_dirichlet"),
                                         ("periodic", "mixed"), ("noslip_noflux", "periodic")])
def test_sides_and_sizes(cdf, m, xcase, ycase):
    sizes = [(6, 6), (7, 64), (33, 17), (64, 64), (65, 31), (130, 9), (39, 77)]
    check(cdf, [_rand_problem(nx, ny, m, 3 * nx + ny, xcase, ycase) for nx, ny in sizes])


def test_small_walled_lattices(cdf):
    check(cdf, [_rand_problem(nx, ny, 2, 5, "mixed", "noslip_noflux")
                for nx, ny in [(1, 1), (9, 1), (1, 9), (2, 2), (3, 200), (200, 3)]])


def test_short_periodic_axis_runs_on_the_persistent_kernel(cdf):
    check(cdf, [_rand_problem(nx, ny, 2, 8, "periodic", "noslip_noflux") for nx, ny in [(5, 20), (40, 12)]])


def test_several_groups(cdf):
    """More instances than one launch takes, enough nodes for the largest tiles, uneven groups."""
    sizes = [(33, 17), (64, 64), (70, 50), (6, 90), (130, 40)]
    check(cdf, [_rand_problem(*sizes[k % 5], 2, k, "mixed", "noslip_noflux") for k in range(70)], steps=(2, 33, 1))
    check(cdf, [_rand_problem(16, 16, 1, k, "periodic", "mixed") for k in range(300)], steps=(34,))
