"""The persistent batch kernel: a lattice with a periodic axis below six nodes has no two-step
tiling and takes the whole batch there, in mode 0.  Several steps a launch (grid barriers, the
source of the step before updated in place), tile shapes and remainders, against the single-lattice
solver, bit for bit; the same on the bounds-checked build.  And which kernel mode 0 runs."""
import os
import subprocess
import sys

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2101_03055_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = [((64, 4), 32), ((32, 8), 7), ((128, 1), 1), ((256, 1), 5)]


def sweep():
    side = I.periodic_side(2)
    narrow = I.chemotaxis_plume(5, 41, seed=8).replace(west=side, east=side)
    return [*I.chemotaxis_plume_sweep(4, seed=3, wmin=16, wmax=140, hmin=9, hmax=70), narrow]


def run_cases(lib):
    out = {}
    for tile, spl in CASES:
        b = lib.BatchSolver(sweep(), tile=tile, steps_per_launch=spl, mode=0)
        assert b.launches(67) == -(-67 // spl)
        b.step(67)
        b.step(3)
        for k in range(5):
            out[f"{tile[0]}x{tile[1]}_{spl}_{k}"] = b.moments(k)
        b.close()
    return out


def test_equals_the_single_lattice_solver(cdf):
    got = run_cases(cdf)
    for k, pb in enumerate(sweep()):
        s = cdf.Solver(pb)
        s.step(70)
        want = s.moments()
        for name in got:
            if name.endswith(f"_{k}"):
                assert np.array_equal(got[name], want), name


def test_checks_build_is_clean(cdf, tmp_path):
    from paper_2101_03055_gb300 import build
    build.build(checks=True)
    path = str(tmp_path / "checks.npz")
    r = subprocess.run([sys.executable, os.path.abspath(__file__), path], env=dict(os.environ, CDF_CHECKS="1"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    got = np.load(path)
    for name, arr in run_cases(cdf).items():
        assert np.array_equal(got[name], arr), name


def test_mode_0_kernels(cdf):
    """Two-step launches of groups where every lattice has the tiling: one for two steps of each group of the four
    small lattices, and one for an odd step."""
    b = cdf.BatchSolver(sweep()[:4], tile=(64, 4), mode=0, steps_per_launch=7)
    groups = b.launches(2)
    assert 1 <= groups <= 4 and b.launches(67) == 33 * groups + 1
    for mode, per_two in ((1, 8), (2, 4)):
        c = cdf.BatchSolver(sweep()[:4], tile=(32, 8), mode=mode, chain_tile_y=6 if mode == 2 else 0)
        assert c.launches(2) == per_two and c.launches(3) == per_two + 4


@pytest.mark.parametrize("m,nx,ny,count,pair", [(2, 2000, 1, 500, False), (4, 2000, 1, 300, False), (2, 64, 64, 40, True),
                                                (4, 3, 2000, 60, True)])
def test_thin_lattices_run_on_the_faster_kernel(cdf, m, nx, ny, count, pair):
    """Rows of one node leave the two-step launches' CTAs mostly idle: 2.2 times the persistent kernel's time with two
    scalars, 3.4 with four; columns of three nodes waste its 128 x 1 tiles: 3.9 times the two-step launches'."""
    from test_parity_gpu import _rand_problem
    pb = _rand_problem(nx, ny, m, 3, "mixed", "noslip_noflux")
    b = cdf.BatchSolver([pb] * count, tile=(128, 1), mode=0, init=False)
    assert (b.launches(64) > 2) == pair
    b.close()


@pytest.mark.parametrize("tile", [(64, 4), None])
@pytest.mark.parametrize("m,nx,ny", [(3, 60, 2), (4, 9, 9), (1, 7, 7), (3, 40, 30)])
def test_timed_batches_keep_the_bits(cdf, tile, m, nx, ny):
    from test_parity_gpu import _rand_problem
    pbs = [_rand_problem(nx, ny, m, 3 + k, "periodic", "noslip_noflux") for k in range(5)]
    b = cdf.BatchSolver(pbs, **(dict(tile=tile, mode=0) if tile else {}))
    b.step(33)
    b.step(2)
    for k, pb in enumerate(pbs):
        s = cdf.Solver(pb)
        s.step(35)
        assert np.array_equal(b.moments(k), s.moments()), k


if __name__ == "__main__":
    from paper_2101_03055_gb300 import lib
    assert lib.CHECKS and lib.cdf_checks_enabled(), "the checks library was not loaded"
    np.savez(sys.argv[1], **run_cases(lib))
