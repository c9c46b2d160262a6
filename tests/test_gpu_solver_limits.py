"""The Poisson solve around the sizes where the direct solver ends, and beyond them.

Its rows (x) and columns (y) end where 16 lines of an axis no longer fit in 227 KB of
shared memory: 1614 and 1709 points, or 830 and 880 where a prime above 13 divides the
length (its pass needs a second buffer); its planes at 1024 (test_gpu_direct.py). Beyond
that multigrid CG solves, in the FP32 of the mixed store with its deepest levels in one
of three ways, so that each plan below takes another:
  32 x 64 x 1032     levels 16x32x516, 8x16x258, 4x8x129: the last solved exactly
  1664 x 64 x 64     ..., 208x8x8, 104x4x4: the last two in one cluster, the last by sweeps
  1664 x 128 x 128   ..., 104x8x8, 52x4x4: the same, the last by its dense inverse
  64 x 64 x 2048     ..., 8x8x256, 4x4x128: level by level
  1617 x 4 x 6       one level (odd rows): the diagonal alone
The first group is held against the eigenvector solution, the second, too large for it,
against its own FP64 residual.
"""
import math

import numpy as np
import pytest

import tests.test_gpu_direct as direct
from tests._cases import bare

pytestmark = pytest.mark.gpu

EPS0 = direct.EPS0
STORES = [(0, 1e-12), (1, 1e-8)]


@pytest.mark.parametrize("precision,rtol", STORES)
@pytest.mark.parametrize("nx,ny,nz", [(342, 4, 6), (512, 4, 6), (1600, 4, 6), (4, 1701, 6), (829, 4, 5), (4, 877, 5),
                                      (1617, 4, 6), (838, 4, 8), (4, 1712, 8)])
def test_long_rows(nx, ny, nz, precision, rtol):
    direct.test_solve_matches_eigenvector_solution(nx, ny, nz, precision, rtol)


@pytest.mark.parametrize("precision,rtol", STORES)
@pytest.mark.parametrize("nx,ny,nz", [(32, 64, 1032), (64, 64, 2048), (1664, 64, 64), (1664, 128, 128)])
def test_deep_multigrid_plans(nx, ny, nz, precision, rtol):
    import paper_2606_05893_gb300 as pkg
    h, phi_c, phi_a = 2.5e-9, -2.0, 3.0 * nz
    wl = bare(nx=nx, ny=ny, nz=nz, h=h, phi_c=phi_c, phi_a=phi_a)
    rho = np.random.default_rng(nx + ny + nz).standard_normal((nz + 1, ny, nx)) * 2e6 + 4e5
    scale = h * h / EPS0
    b = rho[1:nz] * scale
    if precision:
        b = (np.float32(scale) * rho[1:nz].astype(np.float32)).astype(np.float64)
    b[0] += phi_c
    b[-1] += phi_a
    sim = pkg.Simulation(wl, precision=precision, cg_rtol=rtol, cg_maxit=400, preload=False)
    phi, iters, rel = sim.solve(rho)
    sim.close()
    assert rel <= rtol and iters > 0
    assert np.all(phi[0] == phi_c) and np.all(phi[nz] == phi_a)
    x = phi[1:nz]
    r = b - 6.0 * x
    for axis in (1, 2):
        r += np.roll(x, 1, axis) + np.roll(x, -1, axis)
    r[1:] += x[:-1]
    r[:-1] += x[1:]
    # the residual it stops at, and what of it FP64 (12 |x| a node) or float-float cannot tell
    bound = rtol * np.linalg.norm(b) + 12 * np.abs(x).max() * math.sqrt(b.size) * (2.0 ** -46 if precision else 2.0 ** -52)
    assert np.linalg.norm(r) <= bound


@pytest.mark.parametrize("precision", [0, 1])
def test_steps_beyond_the_direct_solver(precision):
    """Recorded steps hold the multigrid CG's loops; their solves converge and count alike without recording."""
    import paper_2606_05893_gb300 as pkg
    wl = bare(nx=32, ny=64, nz=1032, h=2.5e-9, phi_a=500.0, weight=1.0, capacity=1 << 14)
    rng = np.random.default_rng(4)
    wl.preload = [(rng.random((3000, 3)) * np.array(wl.L), rng.standard_normal((3000, 3)) * 1e5) for _ in range(3)]
    rtol = 1e-12 if precision == 0 else 1e-8
    a = pkg.Simulation(wl, precision=precision, cg_rtol=rtol, cg_maxit=400)
    b = pkg.Simulation(wl, precision=precision, cg_rtol=rtol, cg_maxit=400)
    pkg.pic_set_profiling(b.h, True)  # timed steps are always enqueued directly
    a.step(4)
    b.step(4)
    ma, mb = a.moments(), b.moments()
    assert ma["cg_resid_rel"] <= rtol and ma["error_flags"] == 0
    for k in ("count", "abs_cathode", "abs_anode", "next_pid"):
        assert ma[k] == mb[k], k
    a.close()
    b.close()
