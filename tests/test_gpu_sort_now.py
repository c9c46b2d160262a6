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


@pytest.mark.parametrize("precision", [0, 1])
def test_sort_of_one_of_several_instances(precision):
    """An instance of several has a stream of its own: its sort comes after the upload queued on the
    handle's stream, and before the read, the further upload and the ensemble's step that follow."""
    import paper_2606_05893_gb300 as pkg
    rng = np.random.default_rng(9)
    wls = [bare(nx=6, ny=5, nz=8, weight=1e-6, capacity=1 << 17, seed=s, phi_a=1.0) for s in (1, 2)]
    batches = [cloud(rng, wls[0], 60000, 0) for _ in range(3)]
    both = pkg.Simulation(wls, precision=precision, cg_rtol=1e-8)
    alone = pkg.Simulation(wls[1], precision=precision, cg_rtol=1e-8)
    for sim, inst in ((both, 1), (alone, 0)):
        sim.step(2)
        pkg.pic_inject_particles(sim.h, inst, 1, *batches[0])
        sim.sort_now(inst)
        x, _, pid = sim.particles(1, inst)
        cell = np.minimum((x / wls[0].h).astype(int), np.array([5, 4, 7]))
        assert np.array_equal(np.lexsort((pid, (cell[:, 2] * 5 + cell[:, 1]) * 6 + cell[:, 0])), np.arange(60000))
        pkg.pic_inject_particles(sim.h, inst, 1, batches[1][0][:50000], batches[1][1][:50000])
        sim.sort_now(inst)
        sim.step(3)
    a, b = both.moments(1), alone.moments(0)
    for k in ("step", "count", "next_pid", "abs_cathode", "abs_anode", "error_flags"):
        assert a[k] == b[k], k
    (xa, _, pa), (xb, _, pb) = both.particles(1, 1), alone.particles(1, 0)
    assert np.array_equal(xa[np.argsort(pa)], xb[np.argsort(pb)])
    both.close()
    alone.close()
