"""A sort outside a recorded step knows the counts: it does nothing for a species without
particles, and the radix passes of an overfull cell cover the bits of the key that
are in use. The order is (cell, pid) all the same."""
import numpy as np
import pytest

from tests._cases import bare

pytestmark = pytest.mark.gpu


def cloud(rng, wl, n, dense):
    """n particles all over the box and `dense` in one cell."""
    one = (np.array([1, 2, 3]) + 0.05 + 0.9 * rng.random((dense, 3))) * wl.h
    x = np.concatenate([one, rng.random((n, 3)) * np.array(wl.L)])
    return x, rng.standard_normal(x.shape)


def sort_launches(precision, sizes):
    """Launches of one sort of three species of `sizes` = (spread, dense); the first one's order is checked."""
    import paper_2606_05893_gb300 as pkg
    wl = bare(nx=6, ny=5, nz=8, weight=1e-6, capacity=1 << 14)
    rng = np.random.default_rng(7)
    wl.preload = [cloud(rng, wl, *s) for s in sizes]
    sim = pkg.Simulation(wl, precision=precision)
    before = pkg.pic_launch_count()
    sim.sort_now()
    launches = pkg.pic_launch_count() - before
    for sp, (n, dense) in enumerate(sizes):
        start = pkg.pic_get_cell_start(sim.h, 0, sp, 6 * 5 * 8)
        assert start[0] == 0 and start[-1] == n + dense and np.all(np.diff(start) >= 0)
        x, _, pid = sim.particles(sp)
        cell = np.minimum((x / wl.h).astype(int), np.array([5, 4, 7]))
        key = (cell[:, 2] * 5 + cell[:, 1]) * 6 + cell[:, 0]
        assert np.array_equal(np.lexsort((pid, key)), np.arange(n + dense))
    sim.close()
    return launches


@pytest.mark.parametrize("precision", [0, 1])
def test_sort_skips_empty_species(precision):
    every = sort_launches(precision, [(900, 0)] * 3)
    assert sort_launches(precision, [(900, 0), (0, 0), (0, 0)]) <= every // 3 + 2  # a commit each
    assert sort_launches(precision, [(0, 0)] * 3) <= 3


@pytest.mark.parametrize("precision", [0, 1])
def test_radix_passes_cover_the_bits_in_use(precision):
    plain = sort_launches(precision, [(900, 4000), (0, 0), (0, 0)])
    radix = sort_launches(precision, [(900, 5000), (0, 0), (0, 0)])
    bits = (6 * 5 * 8).bit_length() + (5900).bit_length()
    assert 0 < radix - plain <= 1 + 3 * -(-bits // 8)  # the keys, three launches a pass
