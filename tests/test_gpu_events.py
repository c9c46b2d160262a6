"""The order in which a step's events take effect, over the counts where it changes
path: counting by each event's thread (up to 128), runs placed by a block (short
ones, several on a block, the longest, in instances with and without radix passes
in reserve), and the radix passes beyond 131072 events. Every electron ionizes
or finds its cell's neutrals taken, so a step has exactly as many events as
electrons; the log is in the order of effect and must be the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_2606_05893_gb300 import workloads as W
from tests._cases import bare, const_xsec, isotropic, speed_of_eV
from tests.test_gpu_parity import full_compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available()
    import paper_2606_05893_gb300 as p
    p.load_library()
    return p


def crowded(n_e, capacity, seed):
    """n_e electrons, each on an ion, in the middle planes; about as many neutrals in all cells."""
    wl = bare(nx=16, ny=8, nz=8, h=5e-9, dt=1e-16, weight=1.0, capacity=capacity, seed=seed,
              xsec=[const_xsec(W.XS_IONIZATION, 1e-13, threshold=W.CU_IONIZATION_EV)])
    rng = np.random.default_rng(seed)
    xe = np.column_stack([rng.random(n_e) * 16, rng.random(n_e) * 8, 2.0 + rng.random(n_e) * 4]) * wl.h
    ve = isotropic(rng, n_e, speed_of_eV(100.0))
    per = n_e // 512 + 4  # in each of the 1024 cells, whose middle half holds the electrons
    corner = np.stack(np.meshgrid(np.arange(16), np.arange(8), np.arange(8), indexing="ij"), -1).reshape(-1, 3)
    xn = (np.repeat(corner, per, axis=0) + 0.05 + 0.9 * rng.random((1024 * per, 3))) * wl.h
    vn = rng.standard_normal(xn.shape) * 500.0
    wl.preload = [(xe, ve), (xn, vn), (xe.copy(), np.zeros_like(xe))]
    return wl


@pytest.mark.parametrize("n_e,capacity", [(31, 1 << 14), (128, 1 << 14), (129, 1 << 14), (257, 1 << 14), (513, 1 << 20), (4096, 1 << 16),
                                          (5000, 1 << 20), (1 << 17, 1 << 21), (9000, 1 << 22),
                                          (1 << 17, (1 << 21) + 16), ((1 << 17) + 1, (1 << 21) + 16)])
def test_order_of_effect(pkg, n_e, capacity):
    wl = crowded(n_e, capacity, seed=n_e)
    sim = pkg.Simulation(wl, precision=pkg.PIC_FP64, cg_rtol=1e-13, cg_maxit=5000)
    ref = O.Oracle(wl, cg_rtol=1e-13)
    sim.step()
    ref.step()
    mg, _ = full_compare(sim, ref, wl)
    assert mg["n_ionization"] + mg["n_suppressed"] == n_e and mg["n_ionization"] > n_e // 2
    assert np.array_equal(sim.ionization_log(), ref.ionization_log())
    sim.close()
    ref.close()


def test_recorded_radix_passes(pkg):
    """The radix passes as a recorded step holds them, in a node that the step opens by itself: the first
    step (enqueued directly, 131072 events placed by runs) leaves more than 131072 electrons above the
    threshold, and neutrals enough for them, so the recorded ones after it, one of each parity, take the passes."""
    wl = crowded(1 << 17, 1 << 23, seed=77)
    more = [crowded(1 << 17, 1 << 23, seed=78 + q).preload[1] for q in range(4)]
    wl.preload[1] = tuple(np.concatenate(a) for a in zip(wl.preload[1], *more))
    sim = pkg.Simulation(wl, precision=pkg.PIC_FP64, cg_rtol=1e-13, cg_maxit=5000)
    ref = O.Oracle(wl, cg_rtol=1e-13)
    events = 1 << 17
    sim.step()
    ref.step()
    for _ in range(2):
        launches = pkg.pic_launch_count()
        sim.step()
        assert pkg.pic_launch_count() - launches == 1
        ref.step()
        mg, _ = full_compare(sim, ref, wl)
        total = mg["n_ionization"] + mg["n_suppressed"]
        assert total - events > 1 << 17
        events = total
        assert np.array_equal(sim.ionization_log(), ref.ionization_log())
    sim.close()
    ref.close()
