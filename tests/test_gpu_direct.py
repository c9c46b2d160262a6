"""The direct Poisson solver over the sizes where it changes path: every radix of
its FFTs (powers of two, 3 to 13, primes without a butterfly), odd and even rows
(with and without a Nyquist column), rows that do not fill a tile, one to many
warps of planes with ragged last chunks, and the first size beyond it (the
multigrid CG). Reference: the same 7-point problem in FP64 by its eigenvectors
(numpy). The solve stops at ||b - A x|| <= rtol ||b||, so its error is at most
rtol ||b|| / lambda_min, lambda_min = 4 sin^2(pi / (2 nz)) the smallest
eigenvalue; the mixed store solves for the FP32 charge term, which the reference
takes too, and its residual is known to about 2^-46 of its largest term
12 max|x| (float-float), which adds that term's share to the bound.
"""
import math

import numpy as np
import pytest

from tests._cases import bare

pytestmark = pytest.mark.gpu

EPS0 = 8.8541878128e-12
SIZES = [
    (16, 16, 17), (32, 32, 64), (8, 4, 2), (2, 2, 3), (1, 1, 5), (4, 1, 18), (1, 6, 9), (3, 5, 16),
    (7, 9, 33), (11, 13, 34), (26, 22, 15), (34, 46, 20), (17, 19, 35), (40, 36, 90), (24, 20, 34), (15, 14, 257),
    (128, 64, 40), (256, 16, 12), (62, 128, 9), (96, 80, 150), (10, 12, 258), (6, 8, 514), (4, 6, 1025), (8, 8, 1026),
]


def _reference(nx, ny, nz, b):
    k = np.arange(1, nz)
    S = math.sqrt(2.0 / nz) * np.sin(math.pi / nz * k[:, None] * k[None, :])

    def lam(n):
        return 4 * np.sin(math.pi * np.arange(n) / n) ** 2

    f = np.fft.fft2(np.einsum("ab,byx->ayx", S, b))
    f /= (4 * np.sin(math.pi * k / (2 * nz)) ** 2)[:, None, None] + lam(ny)[None, :, None] + lam(nx)[None, None, :]
    return np.einsum("ab,byx->ayx", S, np.fft.ifft2(f).real)


@pytest.mark.parametrize("precision,rtol", [(0, 1e-12), (1, 1e-8)])
@pytest.mark.parametrize("nx,ny,nz", SIZES)
def test_solve_matches_eigenvector_solution(nx, ny, nz, precision, rtol):
    import paper_2606_05893_gb300 as pkg
    h, phi_c, phi_a = 2.5e-9, -2.0, 37.0 * nz
    wl = bare(nx=nx, ny=ny, nz=nz, h=h, phi_c=phi_c, phi_a=phi_a)
    rng = np.random.default_rng(nx + 100 * ny + 10000 * nz)
    rho = rng.standard_normal((nz + 1, ny, nx)) * 2e6 + 4e5
    scale = h * h / EPS0
    charge = rho[1:nz] * scale
    if precision:
        charge = (np.float32(scale) * rho[1:nz].astype(np.float32)).astype(np.float64)
    b = charge.copy()
    b[0] += phi_c
    b[-1] += phi_a
    sim = pkg.Simulation(wl, precision=precision, cg_rtol=rtol, cg_maxit=20000, preload=False)
    for guess in (None, rng.standard_normal(rho.shape) * 10):
        phi, iters, rel = sim.solve(rho, guess)
        assert rel <= rtol and iters > 0
        exact = _reference(nx, ny, nz, b)
        lam_min = 4 * math.sin(math.pi / (2 * nz)) ** 2
        bound = rtol * np.linalg.norm(b)
        bound += 12 * np.abs(exact).max() * math.sqrt(b.size) * (2.0 ** -46 if precision else 2.0 ** -52)
        assert np.linalg.norm(phi[1:nz] - exact) <= bound / lam_min
        assert np.all(phi[0] == phi_c) and np.all(phi[nz] == phi_a)
    sim.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_zero_right_hand_side_gives_zero(precision):
    import paper_2606_05893_gb300 as pkg
    wl = bare(nx=12, ny=10, nz=20, phi_c=0.0, phi_a=0.0)
    sim = pkg.Simulation(wl, precision=precision, cg_rtol=1e-10, preload=False)
    guess = np.random.default_rng(1).standard_normal((21, 10, 12))
    phi, iters, rel = sim.solve(np.zeros((21, 10, 12)), guess)
    assert iters == 0 and rel == 0.0 and np.all(phi == 0.0)
    sim.close()


def test_tiny_potentials_do_not_underflow():
    """The FP64 store's FP32 passes work on a residual scaled to unit size."""
    import paper_2606_05893_gb300 as pkg
    wl = bare(nx=12, ny=10, nz=20, phi_c=0.0, phi_a=0.0)
    sim = pkg.Simulation(wl, precision=0, cg_rtol=1e-12, preload=False)
    rho = np.random.default_rng(2).standard_normal((21, 10, 12))
    big, _, _ = sim.solve(rho)
    small, _, rel = sim.solve(rho * 2.0 ** -300)
    assert rel <= 1e-12 and np.array_equal(small * 2.0 ** 300, big)
    sim.close()


@pytest.mark.parametrize("nx,ny,nz,offset", [(24, 20, 34, 0), (24, 20, 34, 1), (7, 33, 60, 1), (64, 64, 64, 0),
                                             (1, 3, 900, 0), (2, 2, 1030, 0)])
def test_static_solve_on_caller_memory(nx, ny, nz, offset):
    """Caller-owned arrays that start on any double, and the CG beyond the direct solver's planes."""
    import torch
    import paper_2606_05893_gb300 as pkg
    rtol, h, phi_a = 1e-11, 2.5e-9, 37.0 * nz
    n = (nz + 1) * ny * nx
    rho = np.random.default_rng(n).standard_normal((nz + 1, ny, nx)) * 2e6
    rho_dev = torch.zeros(n + 2, dtype=torch.float64, device="cuda")[offset:offset + n]
    phi_dev = torch.zeros(n + 2, dtype=torch.float64, device="cuda")[offset:offset + n]
    rho_dev.copy_(torch.from_numpy(rho.reshape(-1)))
    st, iters, rel = pkg.pic_poisson_solve_static(nx, ny, nz, h, -2.0, phi_a, rho_dev.data_ptr(), phi_dev.data_ptr(), rtol, 100000)
    assert st == pkg.PIC_OK and rel <= rtol and iters > 0
    b = rho[1:nz] * (h * h / EPS0)
    b[0] -= 2.0
    b[-1] += phi_a
    exact = _reference(nx, ny, nz, b)
    phi = phi_dev.cpu().numpy().reshape(nz + 1, ny, nx)
    bound = rtol * np.linalg.norm(b) + 12 * np.abs(exact).max() * math.sqrt(b.size) * 2.0 ** -52
    assert np.linalg.norm(phi[1:nz] - exact) <= bound / (4 * math.sin(math.pi / (2 * nz)) ** 2)
    assert np.all(phi[0] == -2.0) and np.all(phi[nz] == phi_a)


@pytest.mark.parametrize("nx,ny,nz", [(13, 15, 118), (22, 49, 103), (39, 13, 98), (16, 40, 72), (64, 64, 64), (8, 8, 9)])
def test_static_solve_keeps_a_margin(nx, ny, nz):
    """A residual of the direct solver is smooth: it may lie twice as far from the solution as its tolerance
    says, where CG stayed below. So a solve whose tolerance is clear of rounding ends at a tenth of it, and a
    guess that already meets the tolerance is kept as it is."""
    import torch
    import paper_2606_05893_gb300 as pkg
    h, rtol = 2.5e-9, 1e-12
    phi_a = 9.375e9 * nz * h
    rng = np.random.default_rng(nx * ny * nz)
    z, y, x = np.meshgrid(np.arange(nz + 1) / nz, np.arange(ny) / ny - 0.5, np.arange(nx) / nx - 0.5, indexing="ij")
    shape = np.exp(-(x * x + y * y) / 0.08) * (0.3 + np.exp(-4 * z))
    for _ in range(6):
        rho = 0.2 * 9.375e9 * EPS0 / (nz * h) * shape * (0.5 + rng.random() + 0.7 * rng.standard_normal(shape.shape))
        rho_dev, phi_dev = torch.from_numpy(rho).cuda(), torch.zeros(rho.shape, dtype=torch.float64, device="cuda")
        args = (nx, ny, nz, h, -2.0, phi_a, rho_dev.data_ptr(), phi_dev.data_ptr())
        st, iters, rel = pkg.pic_poisson_solve_static(*args, rtol, 100000)
        assert st == pkg.PIC_OK and rel <= 0.1 * rtol
        phi = phi_dev.clone()
        st, iters, again = pkg.pic_poisson_solve_static(*args, rtol, 100000)
        assert st == pkg.PIC_OK and iters == 0 and again == rel and torch.equal(phi, phi_dev)
        phi_dev.zero_()
        st, iters, _ = pkg.pic_poisson_solve_static(*args, rtol, 1)
        assert iters == 1


@pytest.mark.parametrize("precision,rtol,nx,ny,nz", [(0, 1e-12, 30, 66, 135), (0, 1e-12, 30, 84, 106), (0, 1e-12, 22, 48, 73),
                                                     (0, 3e-12, 96, 80, 150), (0, 1e-5, 22, 16, 59), (1, 1e-5, 22, 16, 59)])
def test_solve_keeps_a_margin(precision, rtol, nx, ny, nz):
    """The same of pic_solve, at tolerances that a pass may just meet."""
    import paper_2606_05893_gb300 as pkg
    h = 2.5e-9
    wl = bare(nx=nx, ny=ny, nz=nz, h=h, phi_c=-2.0, phi_a=9.375e9 * nz * h)
    sim = pkg.Simulation(wl, precision=precision, cg_rtol=rtol, cg_maxit=20000, preload=False)
    rng = np.random.default_rng(nx * ny * nz)
    z, y, x = np.meshgrid(np.arange(nz + 1) / nz, np.arange(ny) / ny - 0.5, np.arange(nx) / nx - 0.5, indexing="ij")
    shape = np.exp(-(x * x + y * y) / 0.08) * (0.3 + np.exp(-4 * z))
    for _ in range(4):
        rho = 0.2 * 9.375e9 * EPS0 / (nz * h) * shape * (0.5 + rng.random() + 0.7 * rng.standard_normal(shape.shape))
        phi, iters, rel = sim.solve(rho)
        assert rel <= 0.1 * rtol
        again, more, same = sim.solve(rho, phi.copy())
        assert same <= rtol and (more > 0 or np.array_equal(again, phi))
    sim.close()


def test_static_solve_near_rounding():
    """A smooth density between grounded electrodes: |x| is 1500 |b|, so the residual's rounding comes up to
    common tolerances. Whatever is reached is reported, and a looser tolerance is never missed."""
    import torch
    import paper_2606_05893_gb300 as pkg
    nx, ny, nz = 12, 10, 120
    rho = torch.full((nz + 1, ny, nx), 2e6, dtype=torch.float64, device="cuda")
    reached = []
    for rtol in 10.0 ** -np.arange(6.0, 14.0, 0.25):
        phi = torch.zeros_like(rho)
        st, iters, rel = pkg.pic_poisson_solve_static(nx, ny, nz, 2.5e-9, 0.0, 0.0, rho.data_ptr(), phi.data_ptr(), rtol, 1000)
        assert (st == pkg.PIC_OK) == (rel <= rtol) and iters <= 40
        reached.append(st == pkg.PIC_OK)
    assert reached == sorted(reached, reverse=True) and sum(reached) >= 20
